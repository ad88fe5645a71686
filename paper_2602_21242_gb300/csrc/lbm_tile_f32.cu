// lbm_tile_f32.cu -- instantiation of the several-steps-a-launch tiles for the FP32 form.
#include "lbm_tile.cuh"

OLBM_DEFINE_TILE(1, f32)
