// Tile pass instantiations: programs in the kernel parameters (see the end of kernels_tile.cu).
#define QS_TILE_PARAM
#include "kernels_tile.cu"
