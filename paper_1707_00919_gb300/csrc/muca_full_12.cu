// muca_full_12.cu - sweep kernels for L = 12.
#define MUCA_L 12
#include "muca_full.cuh"
