// The batched step for n = 5 nodes per cell and dimension.
#include "dg_batch_step.cuh"

DGK_INSTANTIATE_BATCH(5)
