// The batched step for n = 3 nodes per cell and dimension.
#include "dg_batch_step.cuh"

DGK_INSTANTIATE_BATCH(3)
