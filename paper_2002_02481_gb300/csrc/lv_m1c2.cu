// Monte Carlo kernels of model 1 (the spot weight linear in ln S), cell mode 2
// (other grids, the cell found by bins).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(1, 2)
