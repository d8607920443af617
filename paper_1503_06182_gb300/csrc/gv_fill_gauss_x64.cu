// Fill kernels of the Gaussian integrand, 64-bit-significand form.
#include "gv_fill_inst.cuh"
GV_DEFINE_FILL_LAUNCHER(launch_fill_gauss, GV_GAUSS, GvX, x64)
