// Entry points of the debug library (libuncomp_debug.so) only: parts of the product that have no entry of their own, for tests.
#ifdef UNCOMP_DEBUG
#include "wide_krylov.cuh"

extern "C" {

// 1 when the wide entropy of an n x n matrix starts with block Lanczos on a device that holds `ctas` of its CTAs at once
int uncomp_debug_krylov_applies(int n, int k, int ctas) { return uncomp::krylov_applies(n, k, ctas) ? 1 : 0; }

}  // extern "C"
#endif
