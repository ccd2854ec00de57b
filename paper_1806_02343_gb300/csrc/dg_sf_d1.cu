// Sum-factorised FP64 kernels, degree 1 (see dg_sf_impl.cuh).
#define DG_SF_DEG 1
#include "dg_sf_impl.cuh"
