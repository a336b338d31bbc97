// Monte Carlo kernels of model 1 (the spot weight linear in ln S), cell mode 0
// (the cell found by a conversion or a binary search).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(1, 0)
