// Monte Carlo kernels of model 3 (the Euler scheme on S with the weight linear in ln S), cell mode 2
// (other grids, the cell found by bins).
#include "lv_mc.cuh"

LV_DEFINE_KERNELS(3, 2)
