// lbm_tile_f16.cu -- instantiation of the several-steps-a-launch tiles for the FP16 form.
#include "lbm_tile.cuh"

OLBM_DEFINE_TILE(2, f16)
