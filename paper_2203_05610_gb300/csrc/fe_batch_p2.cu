// fe_batch_p2.cu -- the batch kernels of second-order meshes
#include "fe_batch_kernel.cuh"

const void* fe_batch_kernel_p2(bool f64, int nt) { return batch_kernel<2>(f64, nt); }

FE_DBG_BOUNDS_READER(fe_dbg_bounds_batch_p2)
