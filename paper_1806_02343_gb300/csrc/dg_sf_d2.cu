// Sum-factorised FP64 kernels, degree 2 (see dg_sf_impl.cuh).
#define DG_SF_DEG 2
#include "dg_sf_impl.cuh"
