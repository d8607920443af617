// Fill kernels of the e+e- -> q qbar g integrand, 64-bit-significand form.
#include "gv_fill_inst.cuh"
GV_DEFINE_FILL_LAUNCHER(launch_fill_ee3j, GV_EE3J, GvX, x64)
