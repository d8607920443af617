// Fill kernels with a histogram of the observable, 64-bit-significand form (all integrands).
#include "gv_fill_inst.cuh"
GV_DEFINE_FILL_HIST_LAUNCHER(GvX, x64)
