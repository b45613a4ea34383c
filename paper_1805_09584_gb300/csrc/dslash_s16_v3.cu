// Compiled launch shape 3 of the sloppy stencil (64 threads per block, 7 resident blocks
// per SM, next-direction prefetch on, 2 right-hand sides per pass): its own translation
// unit so that the shapes compile in parallel.
#include "s16_kernels.cuh"

TMND_S16_DEFINE_SHAPE(3, 64, 7, true, 2)
