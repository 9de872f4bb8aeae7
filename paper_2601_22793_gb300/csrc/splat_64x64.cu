// The splat's tile kernels with 64 x 64 tiles (splat_tile.cuh).
#define EPR_SPLAT_KERNELS
#include "splat_tile.cuh"

EPR_SPLAT_DEFINE(64, 64)
