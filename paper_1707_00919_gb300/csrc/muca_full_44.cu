// muca_full_44.cu - sweep kernels for L = 44.
#define MUCA_L 44
#include "muca_full.cuh"
