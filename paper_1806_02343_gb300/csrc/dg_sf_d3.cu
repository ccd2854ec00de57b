// Sum-factorised FP64 kernels, degree 3 (see dg_sf_impl.cuh).
#define DG_SF_DEG 3
#include "dg_sf_impl.cuh"
