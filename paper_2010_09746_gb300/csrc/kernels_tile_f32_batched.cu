// Tile pass instantiations: complex64, batched launches (see the end of kernels_tile.cu).
#define QS_TILE_F32_BATCHED
#include "kernels_tile.cu"
