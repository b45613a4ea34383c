// The sloppy stencil with a thread per site for both flavours: the form for one right-hand side per launch on
// lattices that fill the chip.
//
// Operator, storage and arithmetic are those of s16_kernels.cuh and s16_hop.cuh, and so is every result, bit for
// bit.  There a tile's links are decoded into shared memory, which pays when several right-hand sides read them;
// with one they are written and read once.  Here a thread decodes a direction's link into registers, and the
// two flavours, which share every link entry, make the pairs of the packed f32x2 instructions (with a flavour's
// two spins as pairs, as there, the lower spins' accumulations do not pack: 0.645 ms where it is 0.637).  One loop
// serves all loop orders: with a copy of the site's code in each, as in walk(), the launches take 0.637 ms instead of
// 0.602.  Qhat^2 + sigma with one right-hand side, tiles and this form: 32^3x64 0.666 -> 0.602 ms, 24^3x48
// 0.227 -> 0.208 ms; the four launches of a sloppy multi-shift iteration 0.688 -> 0.619 and 0.242 -> 0.213 ms,
// 16^3x32 65 -> 57 us.  Below that (16x8^3 24 us) and with several right-hand sides (8 at 24^3x48 1.30 ms, 1.49 in
// this form) the tiles are the faster ones.  168 registers, 12 warps per SM: bound by the FP32 pipe and the
// neighbours' latency together.
#pragma once

#include "launch.cuh"
#include "s16_kernels.cuh"

namespace {

// The f2 below are (flavour 0, flavour 1).
// What one direction needs: the neighbour's words, the link's
struct SiteRaw {
    Raw f[2];
    int l[6];
};
__device__ __forceinline__ void pair_of(const Raw r[2], int k, f2 &re, f2 &im) {  // biased floats of component k
    const int w0 = word(r[0], k), w1 = word(r[1], k);
    re = make_float2(s16_flo(w0), s16_flo(w1));
    im = make_float2(s16_fhi(w0), s16_fhi(w1));
}

template <int P>
struct Nbr {
    int n[8];         // direction 2 mu + (0 forward, 1 backward)
    float sf, sb;     // antiperiodic signs of the time direction
    __device__ __forceinline__ Nbr(const LatGeom &g, int apbc, int h) {
        neighbours<0, P>(g, h, n[0], n[1]);
        neighbours<1, P>(g, h, n[2], n[3]);
        neighbours<2, P>(g, h, n[4], n[5]);
        neighbours<3, P>(g, h, n[6], n[7]);
        sf = apbc && n[0] < h ? -1.0f : 1.0f;
        sb = apbc && n[1] > h ? -1.0f : 1.0f;
    }
};

// Hop of direction MU, DIR into acc[spin][colour][re, im]; sg: the antiperiodic sign.  Projection and
// reconstruction are those of s16_hop.cuh's hop_dir.
template <int MU, int DIR, bool G5IN, bool FIRST>
__device__ __forceinline__ void site_dir(const SiteRaw &r, float sg, f2 acc[4][3][2]) {
    f2 u[9];
    decode_link(r.l, 1.0f, u);
    constexpr bool plus = (DIR < 0) != G5IN;
    constexpr int P = plus ? 1 : -1;
    f2 chr[2][3], chi[2][3];
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const int sl = MU == 0 || MU == 3 ? 2 + s : 3 - s;
            f2 uR, uI, lR, lI;
            pair_of(r.f, s * 3 + c, uR, uI);
            pair_of(r.f, sl * 3 + c, lR, lI);
            if (MU == 0 || (MU == 2 && s == 0)) {
                chr[s][c] = comb<-P, -P>(uR, lR);
                chi[s][c] = comb<-P, -P>(uI, lI);
            } else if (MU == 2) {
                chr[s][c] = comb<P, P>(uR, lR);
                chi[s][c] = comb<P, P>(uI, lI);
            } else if (MU == 1 || s == 0) {
                chr[s][c] = comb<P, P>(uR, lI);
                chi[s][c] = comb<-P, -P>(uI, lR);
            } else {
                chr[s][c] = comb<-P, -P>(uR, lI);
                chi[s][c] = comb<P, P>(uI, lR);
            }
        }
    const float cs = sg * r.f[0].nrm * INV_QMAX;
    const f2 cs2 = dup(cs), ncs2 = dup(-cs);
    const f2 cl2 = DIR > 0 ? ncs2 : cs2, ncl2 = DIR > 0 ? cs2 : ncs2;  // factor of the lower spins, its negative
    f2 vr[2][3], vi[2][3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        f2 wr[3], wa[3], wb[3];
#pragma unroll
        for (int j = 0; j < 3; j++) {
            const f2 w = DIR > 0 ? u[i * 3 + j] : u[j * 3 + i];
            wr[j] = dup(w.x);
            wa[j] = dup(DIR > 0 ? fneg(w.y) : w.y);
            wb[j] = dup(DIR > 0 ? w.y : fneg(w.y));
        }
#pragma unroll
        for (int s = 0; s < 2; s++) {
            f2 a = mul2(wr[0], chr[s][0]);
            a = fma2(wr[1], chr[s][1], a);
            a = fma2(wr[2], chr[s][2], a);
            a = fma2(wa[0], chi[s][0], a);
            a = fma2(wa[1], chi[s][1], a);
            vr[s][i] = fma2(wa[2], chi[s][2], a);
            f2 b = mul2(wr[0], chi[s][0]);
            b = fma2(wr[1], chi[s][1], b);
            b = fma2(wr[2], chi[s][2], b);
            b = fma2(wb[0], chr[s][0], b);
            b = fma2(wb[1], chr[s][1], b);
            vi[s][i] = fma2(wb[2], chr[s][2], b);
        }
    }
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            f2 lr, li, fr, fi;  // added to the lower spin 2 + s: (fr lr, fi li)
            if (MU == 0) { lr = vr[s][c]; li = vi[s][c]; fr = ncl2; fi = ncl2; }
            else if (MU == 1) { lr = vi[1 - s][c]; li = vr[1 - s][c]; fr = ncl2; fi = cl2; }
            else if (MU == 2) { lr = vr[1 - s][c]; li = vi[1 - s][c]; fr = fi = s == 0 ? cl2 : ncl2; }
            else { lr = vi[s][c]; li = vr[s][c]; fr = s == 0 ? ncl2 : cl2; fi = s == 0 ? cl2 : ncl2; }
            if (FIRST) {
                acc[s][c][0] = mul2(cs2, vr[s][c]);
                acc[s][c][1] = mul2(cs2, vi[s][c]);
                acc[s + 2][c][0] = mul2(fr, lr);
                acc[s + 2][c][1] = mul2(fi, li);
            } else {
                acc[s][c][0] = fma2(cs2, vr[s][c], acc[s][c][0]);
                acc[s][c][1] = fma2(cs2, vi[s][c], acc[s][c][1]);
                acc[s + 2][c][0] = fma2(fr, lr, acc[s + 2][c][0]);
                acc[s + 2][c][1] = fma2(fi, li, acc[s + 2][c][1]);
            }
        }
}

template <int P, int D>
__device__ __forceinline__ void load_dir(const S16In &in, const int2 *__restrict__ links, int Vh, int h,
                                         const Nbr<P> &nb, SiteRaw &r) {
    constexpr int par = (D & 1) ? 1 - P : P;
    load_raw2(in, nb.n[D], r.f);
    load_link(links + ((size_t)par * 4 + D / 2) * 3 * Vh, (D & 1) ? nb.n[D] : h, r.l);
}
template <int P, int D, bool G5IN>
__device__ __forceinline__ void site_seq(const S16In &in, const int2 *__restrict__ links, int Vh, int h, const Nbr<P> &nb,
                                         const SiteRaw &cur, f2 acc[4][3][2]) {
    SiteRaw nxt;
    if constexpr (D < 7) load_dir<P, D + 1>(in, links, Vh, h, nb, nxt);
    site_dir<D / 2, (D & 1) ? -1 : 1, G5IN, D == 0>(cur, D == 0 ? nb.sf : D == 1 ? nb.sb : 1.0f, acc);
    if constexpr (D < 7) site_seq<P, D + 1, G5IN>(in, links, Vh, h, nb, nxt, acc);
}
// H psi at site h
template <int P, bool G5IN>
__device__ __forceinline__ void site_hop(const LatGeom &g, int apbc, const S16In &in, const int2 *__restrict__ links, int h,
                                         f2 acc[4][3][2]) {
    const Nbr<P> nb(g, apbc, h);
    SiteRaw r;
    load_dir<P, 0>(in, links, g.Vh, h, nb, r);
    site_seq<P, 0, G5IN>(in, links, g.Vh, h, nb, r, acc);
}

// quantise and store a site
__device__ __forceinline__ void store_pairs(S16Out out, int h, const f2 v[4][3][2]) {
    float m = 0.0f;
#pragma unroll
    for (int k = 0; k < 24; k++) {
        const f2 a = v[k / 6][k / 2 % 3][k % 2];
        m = fmaxf(m, fmaxf(fabsf(a.x), fabsf(a.y)));
    }
    const float sc = m > 0.0f ? S16_QMAX / m : 0.0f;
    out.nrm[s16_ni(h)] = m * INV_QMAX;
    int w[2][12];
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const f2 re = fma2(v[k / 3][k % 3][0], dup(sc), dup(S16_ENC_MAGIC)), im = fma2(v[k / 3][k % 3][1], dup(sc), dup(S16_ENC_MAGIC));
        w[0][k] = __byte_perm(__float_as_int(re.x), __float_as_int(im.x), 0x5410);
        w[1][k] = __byte_perm(__float_as_int(re.y), __float_as_int(im.y), 0x5410);
    }
    int4 *q = out.q + s16_qi(0, h);
#pragma unroll
    for (int j = 0; j < 6; j++) {
        const int *x = w[j / 3] + 4 * (j % 3);
        q[j * S16_BLOCK_SITES] = make_int4(x[0], x[1], x[2], x[3]);
    }
}

// Orders 0 and 1: the block's own run of sites; 2 and 3: grid stride; all right-hand sides of a site in turn.
template <int NT, class F>
__device__ __forceinline__ void site_walk(int Vh, const S16Batch &bt, F &&site) {
    const int chunk = (Vh + gridDim.x - 1) / gridDim.x;
    const bool own = bt.order < 2;
    const int h1 = own ? min(Vh, (int)(blockIdx.x + 1) * chunk) : Vh, st = own ? NT : NT * gridDim.x;
    for (int h = (own ? blockIdx.x * chunk : blockIdx.x * NT) + threadIdx.x; h < h1; h += st)
        for (int k = 0; k < bt.nrhs; k++) {
            if (bt.rdone && bt.rdone[k * bt.rdone_stride]) continue;
            site(h, k);
        }
}

template <bool DAG, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) k_site_even_s16(LatGeom g, int apbc, SiteTermF st, const int2 *__restrict__ links,
                                                          S16In in, S16Out out, const int *done, S16Batch bt) {
    dependent_begin();
    if (done && *done) return;
    const float a = st.kappa2 * st.inv_det, e = a * st.kpp;
    site_walk<NT>(g.Vh, bt, [&](int h, int k) {
        f2 acc[4][3][2];
        site_hop<0, DAG>(g, apbc, s16_at(in, k * bt.stride), links, h, acc);
        f2 o[4][3][2];
#pragma unroll
        for (int s = 0; s < 4; s++) {
            const float b = a * (DAG ? -st.kp : st.kp) * (s < 2 ? 1.0f : -1.0f);
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const f2 pr = acc[s][c][0], pi = acc[s][c][1];
                o[s][c][0] = make_float2(fmaf(a, pr.x, fmaf(b, pi.x, e * pr.y)), fmaf(a, pr.y, fmaf(-b, pi.y, e * pr.x)));
                o[s][c][1] = make_float2(fmaf(a, pi.x, fmaf(-b, pr.x, e * pi.y)), fmaf(a, pi.y, fmaf(b, pr.y, e * pi.x)));
            }
        }
        store_pairs(s16_at(out, k * bt.stride), h, o);
    });
}

// Reduction partials: a flavour's squares in FP32, the site's sum added in FP64 to the thread's own slot of dynamic
// shared memory, [right-hand side][sum][thread].
template <bool DAG, int EPI, int NT, int MB>
__global__ void __launch_bounds__(NT, MB) k_site_odd_s16(LatGeom g, int apbc, SiteTermF st, const int2 *__restrict__ links,
                                                         S16In psi_all, S16In te_all, S16Out out_all, S16EpiArgs ea,
                                                         S16Batch bt) {
    constexpr bool SUMS = EPI == EPI_STORE_NORMS || EPI == EPI_MMS_R;
    constexpr int NQ = EPI == EPI_STORE_NORMS ? 2 : 1;
    extern __shared__ double site_part[];
    __shared__ double red[40];
    dependent_begin();
    if (ea.done && *ea.done) return;
    const int Vh = g.Vh;
    if (SUMS)
        for (int q = 0; q < NQ * bt.nrhs; q++) site_part[q * NT + threadIdx.x] = 0.0;
    const float kp = DAG ? -st.kp : st.kp;
    site_walk<NT>(Vh, bt, [&](int h, int k) {
        f2 acc[4][3][2];
        site_hop<1, false>(g, apbc, s16_at(te_all, k * bt.stride), links, h, acc);
        const S16In psi = s16_at(psi_all, k * bt.stride), aux = s16_at(ea.aux, k * bt.stride);
        const float sigma = (float)(EPI == EPI_MMS_R && ea.per_rhs_sigma ? ea.sigma_k[k] : ea.sigma);
        const float alpha = EPI == EPI_MMS_R ? (float)ea.alpha[(size_t)k * ea.alpha_stride] : 0.0f;
        const f2 sc2 = dup(psi.nrm[s16_ni(h)]);
        const float sa = EPI == EPI_SHIFT || EPI == EPI_MMS_R ? sigma * aux.nrm[s16_ni(h)] : 0.0f;
        const float2 *rin = ea.r_in + k * ea.r_stride + h;  // FP32 planes, touched once per launch (evict first)
        float2 *rout = ea.r + k * ea.r_stride + h;
        f2 s1 = dup(0.0f), s2 = dup(0.0f);
        // 4 components at a time (a 16-byte word per flavour), loads one group ahead: the whole site's p, y and r
        // are never live at once
        int4 pw[3][2], aw[3][2];
        float2 rv[3][4][2];
        auto load = [&](int j) {
#pragma unroll
            for (int f = 0; f < 2; f++) {
                pw[j][f] = psi.q[s16_qi(f * 3 + j, h)];
                if (EPI == EPI_SHIFT || EPI == EPI_MMS_R) aw[j][f] = aux.q[s16_qi(f * 3 + j, h)];
                if (EPI == EPI_MMS_R)
#pragma unroll
                    for (int m = 0; m < 4; m++) rv[j][m][f] = __ldcs(rin + (size_t)(f * 12 + 4 * j + m) * Vh);
            }
        };
        load(0);
#pragma unroll
        for (int j = 0; j < 3; j++) {
            if (j < 2) load(j + 1);
            const int p0[4] = {pw[j][0].x, pw[j][0].y, pw[j][0].z, pw[j][0].w}, p1[4] = {pw[j][1].x, pw[j][1].y, pw[j][1].z, pw[j][1].w};
            const int a0[4] = {aw[j][0].x, aw[j][0].y, aw[j][0].z, aw[j][0].w}, a1[4] = {aw[j][1].x, aw[j][1].y, aw[j][1].z, aw[j][1].w};
#pragma unroll
            for (int m = 0; m < 4; m++) {
                const int q = 4 * j + m, s = q / 3, c = q % 3;
                const f2 nb2 = dup(-S16_DEC_BIAS);
                const f2 pr = mul2(add2(make_float2(s16_flo(p0[m]), s16_flo(p1[m])), nb2), sc2);
                const f2 pi = mul2(add2(make_float2(s16_fhi(p0[m]), s16_fhi(p1[m])), nb2), sc2);
                const float b = s < 2 ? kp : -kp;
                f2 hr = acc[s][c][0], hi = acc[s][c][1];
                if (DAG && s >= 2) {
                    hr = make_float2(-hr.x, -hr.y);
                    hi = make_float2(-hi.x, -hi.y);
                }
                // y = A psi - H t (dag: A(-mu) psi - gamma_5 H t)
                f2 yr = make_float2(fmaf(-b, pi.x, fmaf(-st.kpp, pr.y, pr.x - hr.x)), fmaf(b, pi.y, fmaf(-st.kpp, pr.x, pr.y - hr.y)));
                f2 yi = make_float2(fmaf(b, pr.x, fmaf(-st.kpp, pi.y, pi.x - hi.x)), fmaf(-b, pr.y, fmaf(-st.kpp, pi.x, pi.y - hi.y)));
                if (EPI == EPI_STORE_NORMS) {
                    s1 = fma2(yr, yr, fma2(yi, yi, s1));
                    s2 = fma2(pr, pr, fma2(pi, pi, s2));
                }
                if (EPI == EPI_SHIFT || EPI == EPI_MMS_R) {
                    yr = fma2(dup(sa), add2(make_float2(s16_flo(a0[m]), s16_flo(a1[m])), nb2), yr);
                    yi = fma2(dup(sa), add2(make_float2(s16_fhi(a0[m]), s16_fhi(a1[m])), nb2), yi);
                }
                if (EPI == EPI_MMS_R) {  // r' = r - alpha w
                    const f2 al2 = dup(-alpha);
                    const f2 xr = fma2(al2, yr, make_float2(rv[j][m][0].x, rv[j][m][1].x));
                    const f2 xi = fma2(al2, yi, make_float2(rv[j][m][0].y, rv[j][m][1].y));
                    __stcs(rout + (size_t)q * Vh, make_float2(xr.x, xi.x));
                    __stcs(rout + (size_t)(12 + q) * Vh, make_float2(xr.y, xi.y));
                    s1 = fma2(xr, xr, fma2(xi, xi, s1));
                }
                acc[s][c][0] = yr;
                acc[s][c][1] = yi;
            }
        }
        if (EPI != EPI_MMS_R) store_pairs(s16_at(out_all, k * bt.stride), h, acc);
        if (SUMS) site_part[NQ * k * NT + threadIdx.x] += (double)(s1.x + s1.y);
        if (NQ == 2) site_part[(NQ * k + 1) * NT + threadIdx.x] += (double)(s2.x + s2.y);
    });
    if (SUMS)
        for (int q = 0; q < NQ * bt.nrhs; q++) {
            const double t = block_sum(site_part[q * NT + threadIdx.x], red);
            if (threadIdx.x == 0) ea.part_out[(size_t)q * gridDim.x + blockIdx.x] = t;
            __syncthreads();
        }
}

template <int NT, int MB>
int site_per_sm() {
    int a = 0, b = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&a, k_site_odd_s16<true, EPI_MMS_R, NT, MB>, NT, sizeof(double) * 2 * NT);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_site_even_s16<true, NT, MB>, NT, 0);
    a = a < b ? a : b;
    return a > 0 ? a : 1;
}

template <int NT, int MB>
void launch_site_odd(const Geom &g, const SiteTermF &st, const int2 *links, S16In psi, S16In te, S16Out out, bool dag,
                     HopEpi epi, const S16EpiArgs &ea, cudaStream_t s, const S16Batch &bt, int nb) {
    const int ntile = (g.Vh + NT - 1) / NT;
    static_assert(sizeof(double) * 2 * TMND_MAX_BATCH * NT <= 46 * 1024, "partials fit the default shared memory");
#define TMND_SITE16(D, E)                                                                                       \
    launch_dependent_smem(ntile <= nb, k_site_odd_s16<D, E, NT, MB>, dim3(nb), NT,                          \
                          E == EPI_STORE_NORMS ? sizeof(double) * 2 * bt.nrhs * NT                              \
                                               : E == EPI_MMS_R ? sizeof(double) * bt.nrhs * NT : (size_t)0,   \
                          s, lat_geom(g), g.apbc, st, links, psi, te, out, ea, bt)
    switch (epi) {
        case EPI_STORE: dag ? TMND_SITE16(true, EPI_STORE) : TMND_SITE16(false, EPI_STORE); break;
        case EPI_STORE_NORMS: dag ? TMND_SITE16(true, EPI_STORE_NORMS) : TMND_SITE16(false, EPI_STORE_NORMS); break;
        case EPI_SHIFT: dag ? TMND_SITE16(true, EPI_SHIFT) : TMND_SITE16(false, EPI_SHIFT); break;
        case EPI_MMS_R: dag ? TMND_SITE16(true, EPI_MMS_R) : TMND_SITE16(false, EPI_MMS_R); break;
    }
#undef TMND_SITE16
}

}  // namespace

// the extern entry points of a shape of this form (I, threads T, blocks per SM B)
#define TMND_S16_DEFINE_SITE_SHAPE(I, T, B)                                                                      \
    int s16_per_sm_##I() { return site_per_sm<T, B>(); }                                                     \
    void s16_even_##I(const Geom &g, const SiteTermF &st, const int2 *links, S16In in, S16Out out, bool dag,    \
                      const int *done, cudaStream_t s, const S16Batch &bt, int nb) {                             \
        const int ntile = (g.Vh + T - 1) / T;                                                                    \
        if (dag)                                                                                                 \
            launch_dependent_if(ntile <= nb, k_site_even_s16<true, T, B>, dim3(nb), T, s, lat_geom(g), g.apbc, st, links, in, out, done, bt);  \
        else                                                                                                     \
            launch_dependent_if(ntile <= nb, k_site_even_s16<false, T, B>, dim3(nb), T, s, lat_geom(g), g.apbc, st, links, in, out, done, bt); \
    }                                                                                                            \
    void s16_odd_##I(const Geom &g, const SiteTermF &st, const int2 *links, S16In psi, S16In te, S16Out out,     \
                     bool dag, HopEpi epi, const S16EpiArgs &ea, cudaStream_t s, const S16Batch &bt, int nb) {   \
        launch_site_odd<T, B>(g, st, links, psi, te, out, dag, epi, ea, s, bt, nb);                          \
    }
