// Monte Carlo kernels of model 2 (the Euler scheme on S), cell mode 0
// (the cell found by a conversion or a binary search).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(2, 0)
