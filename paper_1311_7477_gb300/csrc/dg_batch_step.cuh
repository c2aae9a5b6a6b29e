// The batched step of one n, a device function with external linkage that batch_kernel (dg_batch.cu)
// calls: the five of them compile in parallel and are joined by the device linker.  At most 128
// registers, as batch_kernel: two blocks per SM.
#pragma once

#include "dg_kernels.cuh"

namespace dgk {

template <int N>
__device__ bool batch_step_n(BatchSim* S, const BatchGroup& grp, int vrank, unsigned char* smem, double* redd, float* redf,
                             BarrierState* bs) {
  return batch_step_body<N>(S, grp, vrank, smem, redd, redf, bs);
}

}  // namespace dgk

#define DGK_INSTANTIATE_BATCH(N)                                                                               \
  namespace dgk {                                                                                              \
  template __device__ bool batch_step_n<N>(BatchSim*, const BatchGroup&, int, unsigned char*, double*, float*, \
                                           BarrierState*);                                                     \
  }
