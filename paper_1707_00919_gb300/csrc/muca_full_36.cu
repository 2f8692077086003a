// muca_full_36.cu - sweep kernels for L = 36.
#define MUCA_L 36
#include "muca_full.cuh"
