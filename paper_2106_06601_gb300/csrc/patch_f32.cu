// The patch kernel for float elements (see remap_patch.cuh).
#include "remap_patch.cuh"

namespace costa {

cudaError_t launch_patches_f32(const PatchLaunch &a, int kind, cudaStream_t st) {
    return remap::launch_patch_t<float>(a, kind, st);
}

}  // namespace costa
