// Monte Carlo kernels of model 2 (the Euler scheme on S), cell mode 1
// (log-spaced grids).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(2, 1)
