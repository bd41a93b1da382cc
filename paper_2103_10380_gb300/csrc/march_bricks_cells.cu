// march_bricks_cells.cu -- the ray-march kernels that write every sample's
// cell, for FNR_LAYOUT_BRICKS caches: march.cu's template instantiated in a
// translation unit of its own, so the kernel sets compile in parallel.
#define FNR_MARCH_LAUNCHER launch_march_bricks_cells
#define FNR_MARCH_FORM true, true, true
#include "march.cu"
