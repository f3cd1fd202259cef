// The patch kernel for double elements (see remap_patch.cuh).
#include "remap_patch.cuh"

namespace costa {

cudaError_t launch_patches_f64(const PatchLaunch &a, int kind, cudaStream_t st) {
    return remap::launch_patch_t<double>(a, kind, st);
}

}  // namespace costa
