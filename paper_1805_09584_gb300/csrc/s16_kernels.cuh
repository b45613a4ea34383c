// Kernels of the sloppy stencil: FP32 arithmetic on 16-bit storage (the inner operator of
// the mixed-precision solver).  Same operator as the FP64 kernels
// (Sec. 2: even-odd Schur complement of the ND twisted-mass operator):
//   even:  t_e = kappa^2 A^-1 H_eo psi_o        (dag: kappa^2 A(-mu)^-1 H_eo gamma_5 psi_o)
//   odd :  y_o = A psi_o - H_oe t_e             (dag: A(-mu) psi_o - gamma_5 H_oe t_e)
//
// Storage (16-bit word codec of tmnd_internal.cuh: one complex number per word)
//   spinor (per right-hand side): blocks of 8 sites, each 6 planes of int4,
//     plane j holding complex components 4j..4j+3 (component c = flavour*12 +
//     spin*3 + colour), then the sites' dequantisation scales
//     nrm = max|v| / 32767 (s16_qi / s16_ni of tmnd_internal.cuh).  100 B per site.
//   links: 12-real compression, rows 0 and 1 of U at scale 32767 (|u_ij| <= 1),
//     blocks of 8 sites x 3 planes of int2 per direction and parity (s16_li);
//     row 2 is rebuilt as
//     conj(row0 x row1) (det U = +1, Sec. 2: U in SU(3)).  The antiperiodic
//     sign is applied in the kernel, never folded into links.
//
// A block works on tiles of consecutive sites, a thread per site, flavour and one of RP right-hand sides:
// lane bit 4 is the flavour, for RP = 2 bit 3 the right-hand side, the low bits the site.  The tile's eight
// links per site are decoded once, row 2 included, into shared memory as FP32 and serve both flavours and
// every right-hand side; the neighbours' words come straight from global memory (those of the next
// direction are loaded before the current one is processed).  Arithmetic in s16_hop.cuh.
// RP = 2 halves the shared-memory traffic for the links (a warp's 16-byte reads fall on 8 sites, one line,
// instead of 16; with RP = 1 that traffic keeps the L1 data pipe 68 % busy): 7 % faster at 16^3x32 with 8 right-hand
// sides, 2 % slower at 24^3x48, useless for one.
//
// One thread per site for both flavours (s16_site.cuh) decodes and rebuilds the links for every right-hand side (60
// of 225 instructions per direction) at 168 registers, 12 warps per SM.  Four launches of Qhat^2 + sigma, that form
// and this one: 24^3x48 8 right-hand sides 1.47 -> 1.25 ms; 16^3x32 8 0.35 -> 0.28 ms; an iteration of the
// multi-shift solver at 24^3x48 with 8 (the residual update's FP32 planes loaded all at once) 1.60 -> 1.30 ms.  Here:
// FP32 pipe 53 %, issue 55 %, 17 warps per SM.
//
// This header holds the kernel templates; each compiled launch shape is instantiated
// in a translation unit of its own (dslash_s16_v*.cu, built in parallel) through
// TMND_S16_DEFINE_SHAPE; dslash_s16.cu dispatches between them and runs the autotuner.
#pragma once

#include "lattice.cuh"
#include "launch.cuh"
#include "s16_hop.cuh"

namespace {

// Launch shapes the kernels are compiled in: threads per block, resident blocks per SM the register budget is
// cut for, right-hand sides per pass (0: the form of s16_site.cuh, a site per thread).  The
// autotuner times each on the GPU per (lattice, right-hand sides per launch) and keeps the fastest; shape 0 is the
// default.
#define TMND_S16_SHAPE_LIST(X) X(0, 128, 4, 1) X(1, 128, 5, 2) X(2, 64, 8, 2) X(3, 128, 3, 0)

template <int NT, int RP>
struct Tile {
    static constexpr int SITES = NT / (2 * RP);
    LinkTile<SITES> links;
    int nb[8][SITES];  // neighbours, direction 2 mu + (0 forward, 1 backward)
};

// Neighbours and decoded links of the tile that starts at site h0 (output parity P); links of direction d:
// forward from this parity's sites, backward from the other's.
template <int P, int NT, int RP>
__device__ __forceinline__ void load_tile(const LatGeom &g, int apbc, const int2 *__restrict__ links, int h0,
                                          Tile<NT, RP> &t) {
    constexpr int SITES = Tile<NT, RP>::SITES;
    const size_t stride = 3 * (size_t)g.Vh;
    const int2 *Lp = links + (size_t)P * 4 * stride, *Lq = links + (size_t)(1 - P) * 4 * stride;
#pragma unroll
    for (int w = 0; w < 2 / RP; w++) {
        const int item = threadIdx.x + w * NT, i = item % SITES, mu = item / SITES, h = min(h0 + i, g.Vh - 1);
        int hf, hb;
        float sf = 1.0f, sb = 1.0f;
        if (mu == 0) {
            neighbours<0, P>(g, h, hf, hb);
            if (apbc) {  // a hop across the time boundary carries -1
                sf = hf < h ? -1.0f : 1.0f;
                sb = hb > h ? -1.0f : 1.0f;
            }
        } else if (mu == 1) {
            neighbours<1, P>(g, h, hf, hb);
        } else if (mu == 2) {
            neighbours<2, P>(g, h, hf, hb);
        } else {
            neighbours<3, P>(g, h, hf, hb);
        }
        t.nb[2 * mu][i] = hf;
        t.nb[2 * mu + 1][i] = hb;
        f2 u[9];
        int wv[6];
        load_link(Lp + mu * stride, h, wv);
        decode_link(wv, sf, u);
        t.links.put(2 * mu, i, u);
        load_link(Lq + mu * stride, hb, wv);
        decode_link(wv, sb, u);
        t.links.put(2 * mu + 1, i, u);
    }
}

template <int D, bool G5IN, int NT, int RP>
__device__ __forceinline__ void hop_seq(const Tile<NT, RP> &t, int i, const S16In &in, int f, const Raw &cur, f2 up[3][2],
                                        f2 lo[3][2]) {
    Raw nxt;
    if constexpr (D < 7) load_raw(in, f, t.nb[D + 1][i], nxt);
    f2 u[9];
    t.links.get(D, i, u);
    hop_dir<D / 2, (D & 1) ? -1 : 1, G5IN, D == 0>(cur, u, up, lo);
    if constexpr (D < 7) hop_seq<D + 1, G5IN, NT, RP>(t, i, in, f, nxt, up, lo);
}
// H psi at tile site i, flavour f: v[spin*3 + colour]
template <bool G5IN, int NT, int RP>
__device__ __forceinline__ void hop_all(const Tile<NT, RP> &t, int i, const S16In &in, int f, f2 v[12]) {
    f2 up[3][2], lo[3][2];
    Raw r;
    load_raw(in, f, t.nb[0][i], r);
    hop_seq<0, G5IN, NT, RP>(t, i, in, f, r, up, lo);
#pragma unroll
    for (int c = 0; c < 3; c++) {
        v[c] = make_float2(up[c][0].x, up[c][1].x);
        v[3 + c] = make_float2(up[c][0].y, up[c][1].y);
        v[6 + c] = make_float2(lo[c][0].x, lo[c][1].x);
        v[9 + c] = make_float2(lo[c][0].y, lo[c][1].y);
    }
}

// The loop orders over tiles and right-hand sides.  tile(w) prepares a tile (all threads), site(k) does right-hand
// sides k .. k + RP - 1 of it.
template <int RP, class F, class G>
__device__ __forceinline__ void walk(int ntile, const S16Batch &bt, F &&tile, G &&site) {
    const int t0 = (int)((long long)ntile * blockIdx.x / gridDim.x), t1 = (int)((long long)ntile * (blockIdx.x + 1) / gridDim.x);
    auto off = [&](int k) {  // nothing left to do in this group
        bool o = bt.rdone != nullptr;
        for (int q = k; q < k + RP && q < bt.nrhs && o; q++) o = bt.rdone[q * bt.rdone_stride];
        return o;
    };
    const int groups = (bt.nrhs + RP - 1) / RP;
    if (bt.order == 3) {  // grid stride over (tile, right-hand sides) items
        const long items = (long)ntile * groups;
        for (long w = blockIdx.x; w < items; w += gridDim.x) {
            const int k = (int)(w % groups) * RP;
            if (off(k)) continue;
            tile((int)(w / groups));
            site(k);
        }
    } else if (bt.order == 2) {  // grid stride over tiles: all blocks move through the lattice together, so every
                                 // right-hand side's neighbours stay in L2 while the band passes
        for (int w = blockIdx.x; w < ntile; w += gridDim.x) {
            tile(w);
            for (int k = 0; k < bt.nrhs; k += RP)
                if (!off(k)) site(k);
        }
    } else if (bt.order == 1) {  // each group of right-hand sides over the block's own tiles, one after another
        for (int k = 0; k < bt.nrhs; k += RP)
            for (int w = t0; w < t1 && !off(k); w++) {
                tile(w);
                site(k);
            }
    } else {  // the block's own tiles, every right-hand side of a tile before the next
        for (int w = t0; w < t1; w++) {
            tile(w);
            for (int k = 0; k < bt.nrhs; k += RP)
                if (!off(k)) site(k);
        }
    }
}

// A thread's place: flavour, site of the tile, right-hand side of the pass
template <int RP>
struct Place {
    int f, i, q;
    __device__ __forceinline__ Place() {
        const int lane = threadIdx.x & 31;
        f = lane >> 4;
        i = (threadIdx.x >> 5) * (16 / RP) + (lane & (16 / RP - 1));
        q = RP == 2 ? lane >> 3 & 1 : 0;
    }
    // this thread's right-hand side of the pass from k on; on = false (and another's number) if it has nothing to do
    __device__ __forceinline__ int rhs(int k, const S16Batch &bt, bool &on) const {
        if (RP == 1) return k;
        const bool mine = k + q < bt.nrhs && !(bt.rdone && bt.rdone[(k + q) * bt.rdone_stride]);
        on = on && mine;
        return k + q < bt.nrhs ? k + q : k;
    }
};

template <bool DAG, int NT, int MB, int RP>
__global__ void __launch_bounds__(NT, MB) k_hop_even_s16(LatGeom g, int apbc, SiteTermF st, const int2 *__restrict__ links,
                                                         S16In in, S16Out out, const int *done, int ntile,
                                                         S16Batch bt) {
    __shared__ Tile<NT, RP> t;
    dependent_begin();
    if (done && *done) return;
    const Place<RP> pl;
    const int f = pl.f;
    int h = 0;
    auto tile = [&](int w) {
        __syncthreads();  // the previous tile is done with
        load_tile<0, NT, RP>(g, apbc, links, w * Tile<NT, RP>::SITES, t);
        h = w * Tile<NT, RP>::SITES + pl.i;
        __syncthreads();
    };
    // kappa^2 A^-1, per spin sign g A^-1 = [[a - i kp g, kpp], [kpp, a + i kp g]] / det
    const float a = st.kappa2 * st.inv_det, e = a * st.kpp;
    const float b0 = a * (DAG ? -st.kp : st.kp) * (f == 0 ? 1.0f : -1.0f);
    walk<RP>(ntile, bt, tile, [&](int k0) {
        bool on = h < g.Vh;
        const int k = pl.rhs(k0, bt, on);
        f2 p[12], o[12];
        hop_all<DAG, NT, RP>(t, pl.i, s16_at(in, k * bt.stride), f, p);
#pragma unroll
        for (int q = 0; q < 12; q++) {
            const float b = q < 6 ? b0 : -b0;
            const float x = __shfl_xor_sync(0xffffffffu, p[q].x, 16), y = __shfl_xor_sync(0xffffffffu, p[q].y, 16);
            o[q] = make_float2(fmaf(a, p[q].x, fmaf(b, p[q].y, e * x)), fmaf(a, p[q].y, fmaf(-b, p[q].x, e * y)));
        }
        store_site(s16_at(out, k * bt.stride), f, min(h, g.Vh - 1), on, o);
    });
}

// Reduction partials: a site's 48 squares are added in FP32, the sites in FP64: two sites by a shuffle, then in a
// shared slot per (right-hand side, sum, pair of sites).  Of two sums the second flavour's lanes do the second, so
// that both take one FP64 instruction of each kind.  Against FP32 sums over 4 or 8 sites (four launches of an
// iteration, 8 right-hand sides): 32^3x64 4.33 -> 4.23 ms, 24^3x48 1.32 -> 1.30 ms, 16^3x32 298 -> 307 us.
template <bool DAG, int EPI, int NT, int MB, int RP>
__global__ void __launch_bounds__(NT, MB) k_hop_odd_s16(LatGeom g, int apbc, SiteTermF st, const int2 *__restrict__ links,
                                                        S16In psi_all, S16In te_all, S16Out out_all, S16EpiArgs ea,
                                                        int ntile, S16Batch bt) {
    constexpr bool SUMS = EPI == EPI_STORE_NORMS || EPI == EPI_MMS_R;
    constexpr int NQ = EPI == EPI_STORE_NORMS ? 2 : 1, SITES = Tile<NT, RP>::SITES, SLOTS = SITES / 2;
    __shared__ Tile<NT, RP> t;
    __shared__ double part[SUMS ? TMND_MAX_BATCH * NQ * SLOTS : 1];  // [nrhs][NQ][SLOTS]
    dependent_begin();
    if (ea.done && *ea.done) return;
    const Place<RP> pl;
    const int lane = threadIdx.x & 31, f = pl.f, Vh = g.Vh;
    if (SUMS)
        for (int q = threadIdx.x; q < NQ * bt.nrhs * SLOTS; q += NT) part[q] = 0.0;
    int h = 0;
    auto tile = [&](int w) {
        __syncthreads();  // the previous tile is done with
        load_tile<1, NT, RP>(g, apbc, links, w * SITES, t);
        h = w * SITES + pl.i;
        __syncthreads();
    };
    const float kp0 = (DAG ? -st.kp : st.kp) * (f == 0 ? 1.0f : -1.0f);
    // lane bits: 4 flavour, 3 right-hand side (RP = 2) or site, 0..2 site; bit 2 makes the pairs
    const int slot = (threadIdx.x >> 5) * (8 / RP) + (lane & 3) + (RP == 1 ? lane >> 1 & 4 : 0);
    auto add = [&](float a, float b, int k, bool mine) {
        a += __shfl_xor_sync(0xffffffffu, a, 16);
        if (NQ == 2) b += __shfl_xor_sync(0xffffffffu, b, 16);
        double d = (double)(NQ == 2 && f ? b : a);
        d += __shfl_xor_sync(0xffffffffu, d, 4);
        if (mine && !(lane & 4) && f < NQ) part[(NQ * k + f) * SLOTS + slot] += d;
    };
    walk<RP>(ntile, bt, tile, [&](int k0) {
        bool mine = true;
        const int k = pl.rhs(k0, bt, mine);
        const bool on = mine && h < Vh;
        const S16In te = s16_at(te_all, k * bt.stride), psi = s16_at(psi_all, k * bt.stride);
        const int hc = min(h, Vh - 1);
        f2 v[12];
        hop_all<false, NT, RP>(t, pl.i, te, f, v);
        Raw own, oth;
        load_raw(psi, f, hc, own);
        load_raw(psi, 1 - f, hc, oth);
        float s1 = 0.0f, s2 = 0.0f;
        const float sigma = (float)(EPI == EPI_MMS_R && ea.per_rhs_sigma ? ea.sigma_k[k] : ea.sigma);
        Raw ax;
        if (EPI == EPI_SHIFT || EPI == EPI_MMS_R) load_raw(s16_at(ea.aux, k * bt.stride), f, hc, ax);
        const float alpha = EPI == EPI_MMS_R ? (float)ea.alpha[(size_t)k * ea.alpha_stride] : 0.0f;
#pragma unroll
        for (int q = 0; q < 12; q++) {
            // y = A psi - H t (dag: A(-mu) psi - gamma_5 H t)
            const float b = q < 6 ? kp0 : -kp0;
            const f2 p = value(own, q, own.nrm), x = value(oth, q, own.nrm);
            const f2 hp = DAG && q >= 6 ? make_float2(-v[q].x, -v[q].y) : v[q];
            f2 y = make_float2(fmaf(-b, p.y, fmaf(-st.kpp, x.x, p.x - hp.x)), fmaf(b, p.x, fmaf(-st.kpp, x.y, p.y - hp.y)));
            if (EPI == EPI_STORE_NORMS) {
                s1 = fmaf(y.x, y.x, fmaf(y.y, y.y, s1));
                s2 = fmaf(p.x, p.x, fmaf(p.y, p.y, s2));
            }
            if (EPI == EPI_SHIFT || EPI == EPI_MMS_R) {
                const int w = word(ax, q);
                const float sa = sigma * ax.nrm;
                y = make_float2(fmaf(sa, s16_lo(w), y.x), fmaf(sa, s16_hi(w), y.y));
            }
            v[q] = y;
        }
        if (EPI == EPI_MMS_R) {
            // r' = r - alpha w: FP32 planes, touched once per launch (evict first); all loads in flight at once
            const size_t at = (size_t)f * 12 * Vh + hc;
            const float2 *rin = ea.r_in + k * ea.r_stride + at;
            float2 *rout = ea.r + k * ea.r_stride + at;
            float2 r[12];
#pragma unroll
            for (int q = 0; q < 12; q++) r[q] = __ldcs(rin + (size_t)q * Vh);
#pragma unroll
            for (int q = 0; q < 12; q++) {
                const float2 r1 = make_float2(fmaf(-alpha, v[q].x, r[q].x), fmaf(-alpha, v[q].y, r[q].y));
                if (on) __stcs(rout + (size_t)q * Vh, r1);
                s1 = fmaf(r1.x, r1.x, fmaf(r1.y, r1.y, s1));
            }
        }
        if (EPI != EPI_MMS_R) store_site(s16_at(out_all, k * bt.stride), f, hc, on, v);
        if (SUMS) add(on ? s1 : 0.0f, on ? s2 : 0.0f, k, mine);
    });
    if (SUMS) {
        __syncthreads();
        constexpr int G = NT / 16;  // lanes per sum, 16 sums at a time
        for (int w0 = 0; w0 < NQ * bt.nrhs; w0 += 16) {
            const int w = w0 + threadIdx.x / G;
            const bool valid = w < NQ * bt.nrhs;
            double s = 0.0;
            if (valid)
                for (int j = threadIdx.x % G; j < SLOTS; j += G) s += part[w * SLOTS + j];
#pragma unroll
            for (int off = G / 2; off > 0; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
            if (valid && threadIdx.x % G == 0) ea.part_out[(size_t)w * gridDim.x + blockIdx.x] = s;
        }
    }
}

template <int NT, int MB, int RP>
int per_sm_of(int dev) {
    int a = 0, b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_hop_odd_s16<true, EPI_MMS_R, NT, MB, RP>, NT, 0);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_hop_even_s16<true, NT, MB, RP>, NT, 0);
    a = a < b ? a : b;
    (void)dev;
    return a > 0 ? a : 1;
}

template <int NT, int MB, int RP>
void launch_odd_shape(const Geom &g, const SiteTermF &st, const int2 *links, S16In psi, S16In te, S16Out out,
                      bool dag, HopEpi epi, const S16EpiArgs &ea, cudaStream_t s, const S16Batch &bt, int nb) {
    constexpr int SITES = Tile<NT, RP>::SITES;
    const int ntile = (g.Vh + SITES - 1) / SITES;
#define TMND_ODD16(D, E) \
    launch_dependent_if(ntile <= nb, k_hop_odd_s16<D, E, NT, MB, RP>, dim3(nb), NT, s, lat_geom(g), g.apbc, st, links, psi, te, out, ea, ntile, bt)
    if (!dag) {
        switch (epi) {
            case EPI_STORE: TMND_ODD16(false, EPI_STORE); break;
            case EPI_STORE_NORMS: TMND_ODD16(false, EPI_STORE_NORMS); break;
            case EPI_SHIFT: TMND_ODD16(false, EPI_SHIFT); break;
            case EPI_MMS_R: TMND_ODD16(false, EPI_MMS_R); break;
        }
    } else {
        switch (epi) {
            case EPI_STORE: TMND_ODD16(true, EPI_STORE); break;
            case EPI_STORE_NORMS: TMND_ODD16(true, EPI_STORE_NORMS); break;
            case EPI_SHIFT: TMND_ODD16(true, EPI_SHIFT); break;
            case EPI_MMS_R: TMND_ODD16(true, EPI_MMS_R); break;
        }
    }
#undef TMND_ODD16
}

}  // namespace

// Launches overlap with the kernel before them only on lattices with at most a tile per block: where the blocks
// fill the chip for several tiles, the waiting blocks of the next launch cost 2 % (8 right-hand sides, 24^3x48).
// the extern entry points of one compiled shape (I, threads T, blocks per SM B, right-hand sides per pass R)
#define TMND_S16_DEFINE_SHAPE(I, T, B, R)                                                                        \
    int s16_per_sm_##I() { return per_sm_of<T, B, R>(0); }                                                   \
    void s16_even_##I(const Geom &g, const SiteTermF &st, const int2 *links, S16In in, S16Out out, bool dag,    \
                      const int *done, cudaStream_t s, const S16Batch &bt, int nb) {                             \
        const LatGeom lg = lat_geom(g);                                                                          \
        const int sites = T / (2 * R), ntile = (g.Vh + sites - 1) / sites;                                       \
        if (dag)                                                                                                 \
            launch_dependent_if(ntile <= nb, k_hop_even_s16<true, T, B, R>, dim3(nb), T, s, lg, g.apbc, st, links, in, out, done, ntile, bt);  \
        else                                                                                                     \
            launch_dependent_if(ntile <= nb, k_hop_even_s16<false, T, B, R>, dim3(nb), T, s, lg, g.apbc, st, links, in, out, done, ntile, bt); \
    }                                                                                                            \
    void s16_odd_##I(const Geom &g, const SiteTermF &st, const int2 *links, S16In psi, S16In te, S16Out out,     \
                     bool dag, HopEpi epi, const S16EpiArgs &ea, cudaStream_t s, const S16Batch &bt, int nb) {   \
        launch_odd_shape<T, B, R>(g, st, links, psi, te, out, dag, epi, ea, s, bt, nb);                      \
    }
