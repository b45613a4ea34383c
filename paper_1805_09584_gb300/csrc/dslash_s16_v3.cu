// Compiled launch shape 3 of the sloppy stencil (128 threads per block, 3 resident blocks
// per SM, a site per thread): its own translation unit so
// that the shapes compile in parallel.
#include "s16_site.cuh"

TMND_S16_DEFINE_SITE_SHAPE(3, 128, 3)
