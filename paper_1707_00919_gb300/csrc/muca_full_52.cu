// muca_full_52.cu - sweep kernels for L = 52.
#define MUCA_L 52
#include "muca_full.cuh"
