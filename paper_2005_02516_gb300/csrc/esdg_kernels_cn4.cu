// FP64 kernels in the compact form (no operators stored per element) for
// degree N = 4 with the collapsed volume rule (template parameter + 64).
#define ESDG_N (4 + 64)
#define ESDG_FP64_ONLY
#include "esdg_kernels_impl.cuh"
