// Monte Carlo kernels of model 0 (the main reading), cell mode 1
// (log-spaced grids).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(0, 1)
