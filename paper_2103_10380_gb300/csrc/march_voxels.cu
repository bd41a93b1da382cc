// march_voxels.cu -- launcher of the voxel walk (FNR_RENDER_VOXELS; the
// kernel is in march_voxels.cuh) and the instantiations of its plain form.
#include "march_voxels.cuh"

namespace fnr {

cudaError_t launch_march_voxels(const MarchArgs &a, cudaStream_t s) {
    if (a.total_tiles <= 0) return cudaSuccess;
    const bool skip = (a.r.flags & FNR_RENDER_SKIP_EMPTY) != 0u;
    if (a.f[0].cells != nullptr)  // of every view of a launch or of none
        return skip ? launch_march_voxels_skip_cells(a, s) : launch_march_voxels_cells(a, s);
    return skip ? launch_march_voxels_jump(a, s) : launch_voxels_prec<kVoxPlain>(a, s);
}

}  // namespace fnr
