// lbm_tile_f64df.cu -- instantiation of the several-steps-a-launch tiles for the double-word form.
#include "lbm_tile.cuh"

OLBM_DEFINE_TILE(3, f64df)
