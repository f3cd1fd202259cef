// The patch kernel for float2 elements (see remap_patch.cuh).
#include "remap_patch.cuh"

namespace costa {

cudaError_t launch_patches_c64(const PatchLaunch &a, int kind, cudaStream_t st) {
    return remap::launch_patch_t<float2>(a, kind, st);
}

}  // namespace costa
