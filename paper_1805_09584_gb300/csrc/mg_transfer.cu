// Restriction and prolongation of doublet vectors by the aggregation prolongator (Sec. 3, 3.2), FP32, for up
// to 8 right-hand sides per pass over P.
//
//   restriction   out[rhs][b][f][chi nv + k] = sum_i conj(P[b][chi][k][i]) v[rhs][f][chi][i],  i = (site, 6)
//   prolongation  v[rhs][f][chi][i] = sum_k P[b][chi][k][i] c[rhs][b][f][chi nv + k]
//
// For one block and chirality both are a product of P's nv x 6 nsb matrix with 2 nrhs columns (flavours and
// right-hand sides).  With 8 right-hand sides that is 2.4 G complex multiply-adds at 16^3x32 with 24
// vectors, 62 us of the FP32 pipes, against 74 us for the 0.5 GB of P and vectors from HBM: P has to be
// read once for all columns and the products have to come out of registers.  One thread block per (block,
// chirality); a register tile per thread.  Before, each of the 96 output rows gathered the fine vector
// again: restriction 2768 us, prolongation 654 us; now 209 and 184 us (247 and 244
// before P was prefetched into L1).
//
// The fine vectors are planes over half-lattice sites: a block's sites are contiguous only along z, two of
// a parity in a 4-block.  The prolongation therefore writes pairs.  ZPAIR (block extent in z a multiple of
// 4, 16-byte aligned vectors): the sites z and z + 2, one 16-byte store; otherwise two colour components of
// one site, 8 bytes each.
#include "lattice.cuh"

#include "mg_transfer.cuh"

namespace {

constexpr int TR_THREADS = 256;
constexpr int TR_SITES = 32;               // sites per chunk of the restriction
constexpr int TR_ELEMS = TR_SITES * 6;     // elements per chunk: 6 per lane

struct TrGeom {
    int bd[4], nbd[4];
    int X, Y, Zh, Vh, nsb, nv, nblock;
    FastDiv d3, d2, d1, n3, n2, n1;        // by bd[3..1] and nbd[3..1]
};

// First half-index row of block b: coordinates of its corner.
__device__ __forceinline__ int4 corner(const TrGeom &g, int b) {
    const int r3 = fdiv(b, g.n3), r2 = fdiv(r3, g.n2), r1 = fdiv(r2, g.n1);
    return make_int4(r1 * g.bd[0], (r2 - r1 * g.nbd[1]) * g.bd[1], (r3 - r2 * g.nbd[2]) * g.bd[2],
                     (b - r3 * g.nbd[3]) * g.bd[3]);
}
// (parity, half-index) of local site s of the block at corner o
__device__ __forceinline__ void site_of(const TrGeom &g, int4 o, int s, int &par, int &h) {
    const int r3 = fdiv(s, g.d3), r2 = fdiv(r3, g.d2), r1 = fdiv(r2, g.d1);
    const int z = o.w + s - r3 * g.bd[3], y = o.z + r3 - r2 * g.bd[2], x = o.y + r2 - r1 * g.bd[1], t = o.x + r1;
    par = (t + x + y + z) & 1;
    h = ((t * g.X + x) * g.Y + y) * g.Zh + (z >> 1);
}
// Pair p of a block: its elements, and the site and component of the first
template <bool ZPAIR>
__device__ __forceinline__ void pair_of(int p, int &i0, int &i1, int &s, int &c) {
    if (ZPAIR) {  // 12 pairs per 4 sites along z
        const int grp = p / 12, q = p - grp * 12, iz = q >= 6 ? 1 : 0;
        c = q - 6 * iz;
        s = grp * 4 + iz;
        i0 = s * 6 + c;
        i1 = i0 + 12;
    } else {
        i0 = 2 * p;
        i1 = i0 + 1;
        s = i0 / 6;
        c = i0 - 6 * s;
    }
}

__device__ __forceinline__ void prefetch_l1(const void *p) { asm volatile("prefetch.global.L1 [%0];" ::"l"(p)); }

__device__ __forceinline__ void copy_async8(void *dst, const void *src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(d), "l"(src), "r"(valid ? 8 : 0));
}

// Sums over the lanes of N values: halves are exchanged while N is even, so that a lane ends with the
// values base .. of the ones it started with (the same sums, term by term, as a butterfly of each value).
template <int N, int OFF>
__device__ __forceinline__ void lane_sums(float2 *a, int lane, int &base) {
    if constexpr (OFF > 0) {
        const bool up = lane & OFF;
        if constexpr (N % 2 == 0) {
#pragma unroll
            for (int i = 0; i < N / 2; i++) {
                const float2 keep = up ? a[N / 2 + i] : a[i], send = up ? a[i] : a[N / 2 + i];
                a[i].x = keep.x + __shfl_xor_sync(0xffffffffu, send.x, OFF);
                a[i].y = keep.y + __shfl_xor_sync(0xffffffffu, send.y, OFF);
            }
            base += up ? N / 2 : 0;
            lane_sums<N / 2, OFF / 2>(a, lane, base);
        } else {
#pragma unroll
            for (int i = 0; i < N; i++) {
                a[i].x += __shfl_xor_sync(0xffffffffu, a[i].x, OFF);
                a[i].y += __shfl_xor_sync(0xffffffffu, a[i].y, OFF);
            }
            lane_sums<N, OFF / 2>(a, lane, base);
        }
    }
}
__host__ __device__ constexpr int lane_left(int n, int off) { return off == 0 ? n : lane_left(n % 2 == 0 ? n / 2 : n, off / 2); }

// Warp w: rows (vectors) w, w + 8, .. (RK of them) and NC columns, lane l the elements l, l + 32, ..: P comes
// straight from global memory in whole lines, read once; the columns' elements go through shared memory, two
// chunks deep.  The sums run in the order of one warp per output (lane sums, then across lanes), so the
// coarse vectors, which enter TF32 products, do not depend on the tile.
template <int RK, int NC>
__global__ void __launch_bounds__(TR_THREADS, 2) k_restrict(TrGeom g, const float2 *__restrict__ P,
                                                            const float2 *__restrict__ v, float2 *__restrict__ out,
                                                            int nrhs) {
    extern __shared__ __align__(16) float2 sV[];  // [2][NC][TR_ELEMS]
    const int b = blockIdx.x >> 1, chi = blockIdx.x & 1, rhs0 = blockIdx.y * (NC / 2);
    const int ncol = 2 * min(NC / 2, nrhs - rhs0), tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const int len = g.nsb * 6, nchunk = (g.nsb + TR_SITES - 1) / TR_SITES;
    const size_t Vh = g.Vh;
    const float2 *Pb = P + (size_t)blockIdx.x * ((size_t)g.nv * len);
    const int4 o = corner(g, b);
    const int ls = tid / 6, lc = tid - 6 * ls;  // site and component that this thread fetches of a chunk

    auto load = [&](int ch) {
        if (tid < TR_ELEMS) {
            int par, h;
            const bool in = ch * TR_SITES + ls < g.nsb;
            site_of(g, o, in ? ch * TR_SITES + ls : 0, par, h);
            const float2 *src = v + (((size_t)rhs0 * 2 + par) * 24 + chi * 6 + lc) * Vh + h;
            float2 *dst = sV + (ch & 1) * (NC * TR_ELEMS) + tid;
#pragma unroll
            for (int col = 0; col < NC; col++)
                copy_async8(dst + col * TR_ELEMS,
                            src + (col < ncol ? (size_t)((col >> 1) * 48 + (col & 1) * 12) * Vh : 0), in && col < ncol);
        }
        asm volatile("cp.async.commit_group;");
    };

    const float2 *Pr[RK];
#pragma unroll
    for (int r = 0; r < RK; r++) Pr[r] = Pb + (size_t)min(warp + 8 * r, g.nv - 1) * len;
    float2 acc[RK * NC];
#pragma unroll
    for (int i = 0; i < RK * NC; i++) acc[i] = make_float2(0.f, 0.f);
    load(0);
    for (int ch = 0; ch < nchunk; ch++) {
        if (ch + 1 < nchunk) {
            load(ch + 1);
            asm volatile("cp.async.wait_group 1;");
        } else {
            asm volatile("cp.async.wait_group 0;");
        }
        __syncthreads();
        const float2 *cV = sV + (ch & 1) * (NC * TR_ELEMS) + lane;
        // P's part of the next chunk is on its way while this one is worked on (16 warps per SM alone do not
        // cover the latency: half the stalls waited for P)
        const int inext = (ch + 1) * TR_ELEMS + lane;
#pragma unroll
        for (int j = 0; j < TR_ELEMS / 32; j++)
#pragma unroll
            for (int r = 0; r < RK; r++)
                if (inext + j * 32 < len) prefetch_l1(&Pr[r][inext + j * 32]);
#pragma unroll 3
        for (int j = 0; j < TR_ELEMS / 32; j++) {
            const int i = ch * TR_ELEMS + j * 32 + lane;
            float2 a[RK];
#pragma unroll
            for (int r = 0; r < RK; r++) a[r] = i < len ? __ldg(&Pr[r][i]) : make_float2(0.f, 0.f);
#pragma unroll
            for (int col = 0; col < NC; col++) {
                const float2 x = cV[col * TR_ELEMS + j * 32];
#pragma unroll
                for (int r = 0; r < RK; r++) {
                    float2 &y = acc[r * NC + col];
                    y.x = fmaf(a[r].x, x.x, fmaf(a[r].y, x.y, y.x));
                    y.y = fmaf(a[r].x, x.y, fmaf(-a[r].y, x.x, y.y));
                }
            }
        }
        __syncthreads();
    }
    int base = 0;
    lane_sums<RK * NC, 16>(acc, lane, base);
    constexpr int LEFT = lane_left(RK * NC, 16);
    // lanes that hold the same values (steps without an exchange): the lowest writes
    constexpr int SAME = 32 * LEFT / (RK * NC);
    if (lane % SAME) return;
#pragma unroll
    for (int q = 0; q < LEFT; q++) {
        const int i = base + q, r = i / NC, col = i - r * NC, k = warp + 8 * r;
        if (k < g.nv && col < ncol)
            out[(((size_t)(rhs0 + (col >> 1)) * g.nblock + b) * 2 + (col & 1)) * 2 * g.nv + chi * g.nv + k] = acc[q];
    }
}

// NC columns (2 per right-hand side); a thread owns a pair of elements and all columns.
template <int NC, bool ZPAIR>
__global__ void __launch_bounds__(TR_THREADS) k_prolong(TrGeom g, const float2 *__restrict__ P,
                                                        const float2 *__restrict__ in, float2 *__restrict__ v, int nrhs) {
    __shared__ __align__(16) float2 sc[32][NC];
    const int b = blockIdx.x >> 1, chi = blockIdx.x & 1, rhs0 = blockIdx.y * (NC / 2);
    const int nr = min(NC / 2, nrhs - rhs0);
    const int len = g.nsb * 6;
    const size_t Vh = g.Vh;
    for (int i = threadIdx.x; i < g.nv * NC; i += blockDim.x) {
        const int k = i / NC, col = i - k * NC;
        sc[k][col] = col < 2 * nr ? in[(((size_t)(rhs0 + (col >> 1)) * g.nblock + b) * 2 + (col & 1)) * 2 * g.nv +
                                       chi * g.nv + k]
                                  : make_float2(0.f, 0.f);
    }
    __syncthreads();
    const float2 *Pb = P + (size_t)blockIdx.x * ((size_t)g.nv * len);
    const int4 o = corner(g, b);
    for (int p = threadIdx.x; p < len / 2; p += blockDim.x) {
        int i0, i1, s, c, par, h;
        pair_of<ZPAIR>(p, i0, i1, s, c);
        float2 acc[2][NC];
#pragma unroll
        for (int j = 0; j < NC; j++) acc[0][j] = acc[1][j] = make_float2(0.f, 0.f);
        if (p + blockDim.x < len / 2) {  // the next pair's elements on their way
            int n0, n1, ns, nc;
            pair_of<ZPAIR>(p + blockDim.x, n0, n1, ns, nc);
            for (int k = 0; k < g.nv; k++) {
                prefetch_l1(&Pb[(size_t)k * len + n0]);
                if (ZPAIR) prefetch_l1(&Pb[(size_t)k * len + n1]);
            }
        }
        // few columns leave the loads' latency bare: 8 vectors' elements in flight, 4 where the sums need the registers
        // (24 vectors, 16^3x32: 1 right-hand side 128 -> 108 us, 2 126 -> 108 us; 2^4 aggregates, 8 vectors, 16x8^3, 2
        // right-hand sides 23.4 -> 17.4 us, with both changes)
#pragma unroll(NC <= 4 ? 8 : 4)
        for (int k = 0; k < g.nv; k++) {
            const float2 a0 = __ldg(&Pb[(size_t)k * len + i0]), a1 = __ldg(&Pb[(size_t)k * len + i1]);
#pragma unroll
            for (int j = 0; j < NC; j += 2) {
                const float4 w = *(const float4 *)&sc[k][j];
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const float wr = q ? w.z : w.x, wi = q ? w.w : w.y;
                    acc[0][j + q].x = fmaf(a0.x, wr, fmaf(-a0.y, wi, acc[0][j + q].x));
                    acc[0][j + q].y = fmaf(a0.x, wi, fmaf(a0.y, wr, acc[0][j + q].y));
                    acc[1][j + q].x = fmaf(a1.x, wr, fmaf(-a1.y, wi, acc[1][j + q].x));
                    acc[1][j + q].y = fmaf(a1.x, wi, fmaf(a1.y, wr, acc[1][j + q].y));
                }
            }
        }
        site_of(g, o, s, par, h);
        float2 *dst = v + (((size_t)rhs0 * 2 + par) * 24 + chi * 6 + c) * Vh + h;
#pragma unroll
        for (int j = 0; j < NC; j++) {
            if (j >= 2 * nr) break;
            float2 *d = dst + ((size_t)(j >> 1) * 48 + (j & 1) * 12) * Vh;
            if (ZPAIR) {
                *(float4 *)d = make_float4(acc[0][j].x, acc[0][j].y, acc[1][j].x, acc[1][j].y);
            } else {
                d[0] = acc[0][j];
                d[Vh] = acc[1][j];
            }
        }
    }
}

TrGeom tr_geom(const Geom &g, const int bd[4], const int nbd[4], int nsb, int nv, int nblock) {
    TrGeom r;
    for (int i = 0; i < 4; i++) {
        r.bd[i] = bd[i];
        r.nbd[i] = nbd[i];
    }
    r.X = g.X;
    r.Y = g.Y;
    r.Zh = g.Zh;
    r.Vh = g.Vh;
    r.nsb = nsb;
    r.nv = nv;
    r.nblock = nblock;
    r.d3 = fast_div(bd[3]);
    r.d2 = fast_div(bd[2]);
    r.d1 = fast_div(bd[1]);
    r.n3 = fast_div(nbd[3]);
    r.n2 = fast_div(nbd[2]);
    r.n1 = fast_div(nbd[1]);
    return r;
}

template <int RK, int NC>
cudaError_t start_restrict(const TrGeom &g, const float2 *P, const float2 *v, float2 *out, int nrhs, cudaStream_t s) {
    constexpr size_t bytes = sizeof(float2) * 2 * NC * TR_ELEMS;
    if (bytes > 48 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_restrict<RK, NC>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
        if (e != cudaSuccess) return e;
    }
    k_restrict<RK, NC><<<dim3(2 * g.nblock, (nrhs + NC / 2 - 1) / (NC / 2)), TR_THREADS, bytes, s>>>(g, P, v, out, nrhs);
    return cudaGetLastError();
}
// 48 sums per thread are what the registers hold: 16 columns up to 24 vectors, 8 above
template <int RK>
cudaError_t start_restrict(const TrGeom &g, const float2 *P, const float2 *v, float2 *out, int nrhs, cudaStream_t s) {
    if (nrhs <= 2) return start_restrict<RK, 4>(g, P, v, out, nrhs, s);
    if (nrhs <= 4 || RK == 4) return start_restrict<RK, 8>(g, P, v, out, nrhs, s);
    return start_restrict<RK, RK == 4 ? 8 : 16>(g, P, v, out, nrhs, s);
}
template <int NC>
cudaError_t start_prolong(const TrGeom &g, const float2 *P, const float2 *in, float2 *v, int nrhs, bool zpair,
                          cudaStream_t s) {
    const dim3 grid(2 * g.nblock, (nrhs + NC / 2 - 1) / (NC / 2));
    // no more threads than pairs: 2^4 aggregates have 48 (16^3x32, 8 vectors, 8 right-hand sides: blocks of 256
    // 228 us, of 64 185 us)
    const int pairs = g.nsb * 3, threads = pairs < TR_THREADS ? (pairs + 31) & ~31 : TR_THREADS;
    if (zpair) k_prolong<NC, true><<<grid, threads, 0, s>>>(g, P, in, v, nrhs);
    else k_prolong<NC, false><<<grid, threads, 0, s>>>(g, P, in, v, nrhs);
    return cudaGetLastError();
}

bool zpair_ok(const int bd[4], const void *v) { return bd[3] % 4 == 0 && ((uintptr_t)v & 15) == 0; }

}  // namespace

cudaError_t launch_mg_restrict(const Geom &geom, const int bd[4], const int nbd[4], int nsb, int nv, int nblock,
                               const float2 *P, const float2 *v, float2 *out, int nrhs, cudaStream_t s) {
    const TrGeom g = tr_geom(geom, bd, nbd, nsb, nv, nblock);
    switch ((nv + 7) / 8) {
        case 1: return start_restrict<1>(g, P, v, out, nrhs, s);
        case 2: return start_restrict<2>(g, P, v, out, nrhs, s);
        case 3: return start_restrict<3>(g, P, v, out, nrhs, s);
        default: return start_restrict<4>(g, P, v, out, nrhs, s);
    }
}

cudaError_t launch_mg_prolong(const Geom &geom, const int bd[4], const int nbd[4], int nsb, int nv, int nblock,
                              const float2 *P, const float2 *in, float2 *v, int nrhs, cudaStream_t s) {
    const TrGeom g = tr_geom(geom, bd, nbd, nsb, nv, nblock);
    const bool z = zpair_ok(bd, v);
    if (nrhs == 1) return start_prolong<2>(g, P, in, v, nrhs, z, s);
    if (nrhs == 2) return start_prolong<4>(g, P, in, v, nrhs, z, s);
    if (nrhs <= 4) return start_prolong<8>(g, P, in, v, nrhs, z, s);
    return start_prolong<16>(g, P, in, v, nrhs, z, s);
}
