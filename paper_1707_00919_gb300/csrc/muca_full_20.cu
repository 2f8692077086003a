// muca_full_20.cu - sweep kernels for L = 20.
#define MUCA_L 20
#include "muca_full.cuh"
