// muca_full_4.cu - sweep kernels for L = 4.
#define MUCA_L 4
#include "muca_full.cuh"
