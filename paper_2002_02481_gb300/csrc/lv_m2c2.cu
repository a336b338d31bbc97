// Monte Carlo kernels of model 2 (the Euler scheme on S), cell mode 2
// (other grids, the cell found by bins).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(2, 2)
