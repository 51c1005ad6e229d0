// Tile pass instantiations: complex128 in double-float, batched launches (see the end of kernels_tile.cu).
#define QS_TILE_DF_BATCHED
#include "kernels_tile.cu"
