// Batched fill kernels: GvX, at most 16 axes (4 and 8 events per thread).
#include "gv_fill_batch.cuh"
GV_DEFINE_FILL_BATCH(x16, GvX, 16)
