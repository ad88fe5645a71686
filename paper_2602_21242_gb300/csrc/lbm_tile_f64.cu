// lbm_tile_f64.cu -- instantiation of the several-steps-a-launch tiles for the FP64 form.
#include "lbm_tile.cuh"

OLBM_DEFINE_TILE(0, f64)
