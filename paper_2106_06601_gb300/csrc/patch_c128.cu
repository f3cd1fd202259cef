// The patch kernel for double2 elements (see remap_patch.cuh).
#include "remap_patch.cuh"

namespace costa {

cudaError_t launch_patches_c128(const PatchLaunch &a, int kind, cudaStream_t st) {
    return remap::launch_patch_t<double2>(a, kind, st);
}

}  // namespace costa
