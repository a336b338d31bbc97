// Monte Carlo kernels of model 0 (the main reading), cell mode 0
// (the cell found by a conversion or a binary search).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(0, 0)
