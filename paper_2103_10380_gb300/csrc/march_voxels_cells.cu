// march_voxels_cells.cu -- the voxel walk's instantiations that write every
// walked cell (march_voxels.cuh), compiled apart from the others.
#include "march_voxels.cuh"

namespace fnr {

cudaError_t launch_march_voxels_cells(const MarchArgs &a, cudaStream_t s) { return launch_voxels_prec<kVoxCells>(a, s); }

}  // namespace fnr
