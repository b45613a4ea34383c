// Restriction and prolongation of doublet vectors (mg_transfer.cu).
#pragma once

#include "tmnd_internal.cuh"

cudaError_t launch_mg_restrict(const Geom &geom, const int bd[4], const int nbd[4], int nsb, int nv, int nblock,
                               const float2 *P, const float2 *v, float2 *out, int nrhs, cudaStream_t s);
cudaError_t launch_mg_prolong(const Geom &geom, const int bd[4], const int nbd[4], int nsb, int nv, int nblock,
                              const float2 *P, const float2 *in, float2 *v, int nrhs, cudaStream_t s);
