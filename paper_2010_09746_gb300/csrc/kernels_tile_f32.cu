// Tile pass instantiations: complex64 (see the end of kernels_tile.cu).
#define QS_TILE_F32
#include "kernels_tile.cu"
