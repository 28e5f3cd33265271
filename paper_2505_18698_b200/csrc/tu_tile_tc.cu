// Translation unit of tile_tc.cuh: defines what that header only declares elsewhere.
#define MA_TU_TILE_TC
#include "tile_tc.cuh"
