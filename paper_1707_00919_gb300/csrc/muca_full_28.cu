// muca_full_28.cu - sweep kernels for L = 28.
#define MUCA_L 28
#include "muca_full.cuh"
