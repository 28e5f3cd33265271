// Translation unit of tensor_chain.cuh: defines what that header only declares elsewhere.
#define MA_TU_TENSOR_CHAIN
#include "tensor_chain.cuh"
