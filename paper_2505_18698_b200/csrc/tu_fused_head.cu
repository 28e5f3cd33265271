// Translation unit of fused_head.cuh: defines what that header only declares elsewhere.
#define MA_TU_FUSED_HEAD
#include "fused_head.cuh"
