// Monte Carlo kernels of model 3 (the Euler scheme on S with the weight linear in ln S), cell mode 1
// (log-spaced grids).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(3, 1)
