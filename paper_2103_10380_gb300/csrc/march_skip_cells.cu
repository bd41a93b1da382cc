// march_skip_cells.cu -- the ray-march kernels that write every sample's cell,
// with empty-space skipping: march.cu's template instantiated in a translation
// unit of its own, so the kernel sets compile in parallel.
#define FNR_MARCH_LAUNCHER launch_march_skip_cells
#define FNR_MARCH_FORM true, false, true
#include "march.cu"
