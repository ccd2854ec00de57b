// Specialised Powell kernels of octree meshes and the timestep's face jumps, FP64 degree 2
// (see dg_fast_impl.cuh; uniform meshes run dg_sf_impl.cuh).
#define DG_FAST_T double
#define DG_FAST_DEG 2
#define DG_FAST_CONST 1
#define DG_FAST_UNIFORM 0
#include "dg_fast_impl.cuh"
