// Tile pass instantiations: complex128 in double-float (see the end of kernels_tile.cu).
#define QS_TILE_DF
#include "kernels_tile.cu"
