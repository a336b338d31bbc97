// Monte Carlo kernels of model 0 (the main reading), cell mode 2
// (other grids, the cell found by bins).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(0, 2)
