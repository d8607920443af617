// Batched fill kernels: GvX, at most 4 axes (4 and 8 events per thread).
#include "gv_fill_batch.cuh"
GV_DEFINE_FILL_BATCH(x4, GvX, 4)
