// Monte Carlo kernels of model 1 (the spot weight linear in ln S), cell mode 1
// (log-spaced grids).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(1, 1)
