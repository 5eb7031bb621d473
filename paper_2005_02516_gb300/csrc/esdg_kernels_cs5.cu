// FP64 kernels in the compact form (no operators stored per element) for
// degree N = 5 with the symmetric volume rule (template parameter + 64).
#define ESDG_N (5 + 8 + 64)
#define ESDG_FP64_ONLY
#include "esdg_kernels_impl.cuh"
