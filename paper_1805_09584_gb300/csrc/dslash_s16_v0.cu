// Compiled launch shape 0 of the sloppy stencil (128 threads per block, 4 resident blocks
// per SM, 1 right-hand side per pass): its own translation
// unit so that the shapes compile in parallel.
#include "s16_kernels.cuh"

TMND_S16_DEFINE_SHAPE(0, 128, 4, 1)
