// march_skip.cu -- the ray-march kernels with empty-space skipping
// (FNR_RENDER_SKIP_EMPTY): march.cu's template instantiated with SKIP = true
// in a translation unit of its own, so the kernel sets compile in parallel.
#define FNR_MARCH_LAUNCHER launch_march_skip
#define FNR_MARCH_FORM true, false, false
#include "march.cu"
