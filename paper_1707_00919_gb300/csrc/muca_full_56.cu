// muca_full_56.cu - sweep kernels for L = 56.
#define MUCA_L 56
#include "muca_full.cuh"
