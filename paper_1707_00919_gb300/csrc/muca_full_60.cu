// muca_full_60.cu - sweep kernels for L = 60.
#define MUCA_L 60
#include "muca_full.cuh"
