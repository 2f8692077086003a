// muca_full_40.cu - sweep kernels for L = 40.
#define MUCA_L 40
#include "muca_full.cuh"
