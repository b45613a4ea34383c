// The even-odd reduced operator on FP64-accurate two-digit fixed-point data (hop_fx.cuh), by
// integer multiply-adds.
//
//   even kernel:  t_e = kappa^2 A^-1 H_eo psi_o        (dag: kappa^2 A(-mu)^-1 H_eo gamma_5 psi_o)
//   odd  kernel:  y_o = A psi_o - H_oe t_e             (dag: A(-mu) psi_o - gamma_5 H_oe t_e)
//
// H psi(x) = sum_mu (1 - gamma_mu) U_mu(x) psi(x+mu) + (1 + gamma_mu) U_mu(x-mu)^+ psi(x-mu)
// (Sec. 2, Eq. "Wilson" in the hopping normalisation).  In the chiral basis
// gamma_mu = [[0, B_mu],[B_mu^+, 0]] with B_0 = -1, B_k = -i sigma_k, so
//   (1 - gamma_mu) psi = (chi, -B^+ chi),  chi = psi_up - B psi_lo
//   (1 + gamma_mu) psi = (chi,  B^+ chi),  chi = psi_up + B psi_lo
// and only the two-spin chi is multiplied by the link (spin projection).
//
// Work split.  1152 FP64 multiply-adds per site take 576 clocks of an SM's FP64 pipe; as 3456 integer ones
// they take 115, near the 100 that a site's ~2100 bytes take at the HBM rate.  A block of four warps works
// on 16 sites: warp mu does the two hops of direction mu for both flavours (lanes 0..15 and 16..31), the
// parts meet in shared memory, and warp s finishes spin s.  Against one thread per site and flavour for
// all eight hops this needs no more than 96 registers (five blocks per SM instead of four, no spills to
// speak of), keeps the unrolled link products to one copy per hop sense (the eight copies of the other
// form overran the instruction cache), and is four times shorter for lattices that do not fill the chip.
// Measured for Qhat^2 + sigma (FP64 pipe before, now): 4^4 268 -> 31 us, 16^3x32 934 -> 249 us, 32^3x64
// 13.6 -> 3.48 ms.  What bounds it now: latency and issue together (issue slots 45 %, integer
// multiply-add pipe 60 %, DRAM 25-35 %).
#include <math.h>

#include "hop_fx.cuh"
#include "launch.cuh"
#include "lattice.cuh"

namespace {

// Spin projection of one flavour of a neighbour (in: its first word) for direction MU: digits of
// chi = up -+ B lo, or of its complex conjugate for the backward hop (see hop_run).  G5IN: the input is
// gamma_5 psi.
template <int MU, int DIR, bool G5IN>
__device__ __forceinline__ void project(const int4 *in, int ch[2][3][2], int cl[2][3][2]) {
    constexpr bool plus = (DIR < 0) != G5IN;   // sign of B psi_lo in chi
    constexpr bool swap = MU == 1 || MU == 2;  // B connects spin s with lower spin 1 - s
    constexpr bool imag = MU == 1 || MU == 3;
#pragma unroll
    for (int s = 0; s < 2; s++) {
        // B psi_lo = ph psi_lo[sl]: ph = -1 (mu 0), -i (1), -1 / +1 for s = 0 / 1 (2), -i / +i (3)
        const int sl = swap ? 1 - s : s;
        const bool neg = MU == 2 || MU == 3 ? s == 0 : true;
        const bool sub = neg == plus;  // chi = up -+ (lo or i lo), i lo = (-lo.im, lo.re)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const int4 a = in[(s * 3 + c) * FX_RUN];
            const int4 b = in[((2 + sl) * 3 + c) * FX_RUN];
            ch[s][c][0] = imag ? (sub ? a.x + b.z : a.x - b.z) : (sub ? a.x - b.x : a.x + b.x);
            cl[s][c][0] = imag ? (sub ? a.y + b.w : a.y - b.w) : (sub ? a.y - b.y : a.y + b.y);
            const int ih = imag ? (sub ? a.z - b.x : a.z + b.x) : (sub ? a.z - b.z : a.z + b.z);
            const int il = imag ? (sub ? a.w - b.y : a.w + b.y) : (sub ? a.w - b.w : a.w + b.w);
            ch[s][c][1] = DIR > 0 ? ih : -ih;
            cl[s][c][1] = DIR > 0 ? il : -il;
        }
    }
}

// v = M chi >> d, M the link (DIR > 0) or its transpose.  72 integer multiply-adds per colour component;
// this is the code that all mu share.
template <int DIR>
__device__ __forceinline__ void link_times(const int4 *__restrict__ U, int d, const int ch[2][3][2],
                                           const int cl[2][3][2], long long v[2][3][2]) {
#pragma unroll
    for (int i = 0; i < 3; i++) {
        int4 u[3];
        int nh[3], nl[3];  // the negated imaginary part
#pragma unroll
        for (int j = 0; j < 3; j++) {
            u[j] = __ldg(&U[(DIR > 0 ? i * 3 + j : j * 3 + i) * FX_RUN]);
            nh[j] = -u[j].z;
            nl[j] = -u[j].w;
        }
        // cross terms first (with the half of rounding), then the h h terms on top of their carried-over
        // part; four chains (two spins, real and imaginary part) run side by side
        const long long half = 1ll << 27;
        long long x[2][2] = {{half, half}, {half, half}};
#pragma unroll
        for (int j = 0; j < 3; j++) {
#pragma unroll
            for (int s = 0; s < 2; s++) {
                x[s][0] += (long long)u[j].x * cl[s][j][0];
                x[s][1] += (long long)u[j].x * cl[s][j][1];
            }
#pragma unroll
            for (int s = 0; s < 2; s++) {
                x[s][0] += (long long)u[j].y * ch[s][j][0];
                x[s][1] += (long long)u[j].y * ch[s][j][1];
            }
#pragma unroll
            for (int s = 0; s < 2; s++) {
                x[s][0] += (long long)nh[j] * cl[s][j][1];
                x[s][1] += (long long)u[j].z * cl[s][j][0];
            }
#pragma unroll
            for (int s = 0; s < 2; s++) {
                x[s][0] += (long long)nl[j] * ch[s][j][1];
                x[s][1] += (long long)u[j].w * ch[s][j][0];
            }
        }
#pragma unroll
        for (int s = 0; s < 2; s++) {
            x[s][0] >>= 28;
            x[s][1] >>= 28;
        }
#pragma unroll
        for (int j = 0; j < 3; j++) {
#pragma unroll
            for (int s = 0; s < 2; s++) {
                x[s][0] += (long long)u[j].x * ch[s][j][0];
                x[s][1] += (long long)u[j].x * ch[s][j][1];
            }
#pragma unroll
            for (int s = 0; s < 2; s++) {
                x[s][0] += (long long)nh[j] * ch[s][j][1];
                x[s][1] += (long long)u[j].z * ch[s][j][0];
            }
        }
#pragma unroll
        for (int s = 0; s < 2; s++) {
            v[s][i][0] = x[s][0] >> d;
            v[s][i][1] = x[s][1] >> d;
        }
    }
}

// What the four warps of a block exchange per run of 16 sites
struct FxShared {
    long long part[4][4][3][2][32];  // [direction][forward + backward, backward - forward][...][lane]
    int e[4][32];                    // exponent of each direction's part
    unsigned oh[4][32], ol[4][32];   // leading bits of each spin's sum
};

// Sum of one spin over the directions from the parts in shared memory.  Spins 0, 1: the sums
// forward + backward; spins 2, 3: B^+ (backward - forward).
template <int SPIN>
__device__ __forceinline__ int hop_sum(const FxShared &sm, int spin, long long v[3][2]) {
    const int lane = threadIdx.x & 31;
    int e[4];
#pragma unroll
    for (int m = 0; m < 4; m++) e[m] = sm.e[m][lane];
    const int em = max(max(e[0], e[1]), max(e[2], e[3]));
#pragma unroll
    for (int m = 0; m < 4; m++) {
        const int d = min(em - e[m], 63);
        if (SPIN < 2) {
#pragma unroll
            for (int c = 0; c < 3; c++)
#pragma unroll
                for (int k = 0; k < 2; k++) {
                    const long long t = sm.part[m][spin][c][k][lane] >> d;
                    v[c][k] = m == 0 ? t : v[c][k] + t;
                }
        } else {
            // B^+ w to spin l from spin sl: -1 (mu 0), i (1), +1 / -1 for l = 0 / 1 (2), i / -i (3)
            constexpr int l = SPIN - 2;
            const int sl = m == 1 || m == 2 ? 1 - l : l;
            const bool neg = m == 0 || (m >= 2 && l == 1), imag = m == 1 || m == 3;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const long long wr = sm.part[m][2 + sl][c][0][lane] >> d, wi = sm.part[m][2 + sl][c][1][lane] >> d;
                const long long tr = imag ? (neg ? wi : -wi) : (neg ? -wr : wr);
                const long long ti = imag ? (neg ? -wr : wr) : (neg ? -wi : wi);
                v[c][0] = m == 0 ? tr : v[c][0] + tr;
                v[c][1] = m == 0 ? ti : v[c][1] + ti;
            }
        }
    }
    return em;
}

// H applied to one run of 16 sites (h: the lane's site, of parity P) by a block of four warps.  Warp mu
// takes direction mu, then adds up the four directions of spin mu: v 2^(e - 56), |v| <= 2^61.3, with the
// flavour of the lane's half.  Returns e, the largest exponent among the neighbours.
template <int P, bool G5IN>
__device__ __forceinline__ int hop_run(const LatGeom &g, const int4 *__restrict__ links, const int4 *in,
                                       const int *ex, int h, FxShared &sm, long long v[3][2]) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int nb[2];
    switch (w) {
        case 0: neighbours<0, P>(g, h, nb[0], nb[1]); break;
        case 1: neighbours<1, P>(g, h, nb[0], nb[1]); break;
        case 2: neighbours<2, P>(g, h, nb[0], nb[1]); break;
        default: neighbours<3, P>(g, h, nb[0], nb[1]);
    }
    const int ef = ex[nb[0]], eb = ex[nb[1]], em = max(ef, eb);
    const size_t mu_stride = 9 * fx_sites(g.Vh);
    const int4 *qf = in + fx_at(nb[0], 24), *qb = in + fx_at(nb[1], 24);
    const int4 *uf = links + ((size_t)P * 4 + w) * mu_stride + fx_at(h, 9);
    const int4 *ub = links + ((size_t)(1 - P) * 4 + w) * mu_stride + fx_at(nb[1], 9);
    // the backward hop's words on their way to L1 while the forward hop is worked on
#pragma unroll
    for (int c = 0; c < 12; c++) asm volatile("prefetch.global.L1 [%0];" ::"l"(qb + c * FX_RUN));
#pragma unroll
    for (int c = 0; c < 9; c++) asm volatile("prefetch.global.L1 [%0];" ::"l"(ub + c * FX_RUN));
    long long x[2][3][2], y[2][3][2];
    {  // forward: U chi
        int ch[2][3][2], cl[2][3][2];
        switch (w) {
            case 0: project<0, +1, G5IN>(qf, ch, cl); break;
            case 1: project<1, +1, G5IN>(qf, ch, cl); break;
            case 2: project<2, +1, G5IN>(qf, ch, cl); break;
            default: project<3, +1, G5IN>(qf, ch, cl);
        }
        link_times<+1>(uf, min(em - ef, 63), ch, cl, x);
    }
    {  // backward: U^+ chi = conj(U^T conj(chi))
        int ch[2][3][2], cl[2][3][2];
        switch (w) {
            case 0: project<0, -1, G5IN>(qb, ch, cl); break;
            case 1: project<1, -1, G5IN>(qb, ch, cl); break;
            case 2: project<2, -1, G5IN>(qb, ch, cl); break;
            default: project<3, -1, G5IN>(qb, ch, cl);
        }
        link_times<-1>(ub, min(em - eb, 63), ch, cl, y);
    }
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            sm.part[w][s][c][0][lane] = x[s][c][0] + y[s][c][0];
            sm.part[w][s][c][1][lane] = x[s][c][1] - y[s][c][1];
            sm.part[w][2 + s][c][0][lane] = y[s][c][0] - x[s][c][0];
            sm.part[w][2 + s][c][1][lane] = -y[s][c][1] - x[s][c][1];
        }
    sm.e[w][lane] = em;
    __syncthreads();
    switch (w) {
        case 0:
        case 1: return hop_sum<0>(sm, w, v);
        case 2: return hop_sum<2>(sm, w, v);
        default: return hop_sum<3>(sm, w, v);
    }
}

// Common left shift that brings the largest of the site's 48 words (each below 2^62) to bit 61; 64 if all
// are zero.
__device__ __forceinline__ int norm_shift(const long long v[3][2], FxShared &sm) {
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    unsigned oh = 0, ol = 0;
#pragma unroll
    for (int c = 0; c < 3; c++)
#pragma unroll
        for (int k = 0; k < 2; k++) {
            const int hi = (int)(v[c][k] >> 32);
            oh |= (unsigned)(hi ^ (hi >> 31));
            ol |= (unsigned)v[c][k] ^ (unsigned)(hi >> 31);
        }
    // (a negative word v counts as -v - 1, a place short for -2^k: the bounds have room for it)
    sm.oh[w][lane] = oh;
    sm.ol[w][lane] = ol;
    __syncthreads();
    oh = ol = 0;
#pragma unroll
    for (int k = 0; k < 4; k++) {
        oh |= sm.oh[k][lane] | sm.oh[k][lane ^ 16];
        ol |= sm.ol[k][lane] | sm.ol[k][lane ^ 16];
    }
    return oh ? __clz(oh) - 2 : ol ? 30 + __clz(ol) : 64;
}

// digits of (v << L) / 64, |v << L| <= 2^62
__device__ __forceinline__ void norm_split(long long v, int L, int &h, int &l) {
    const long long t = (v << L) + (32ll + (1ll << 33));
    h = (int)(t >> 34);
    l = ((int)(t >> 6) & 0x0fffffff) - (1 << 27);
}

// (a + b c + ...) of digit products: x += cross terms, y += h h terms
__device__ __forceinline__ void mac(int2 c, int h, int l, long long &x, long long &y) {
    x += (long long)c.x * l;
    x += (long long)c.y * h;
    y += (long long)c.x * h;
}

// A block of four warps takes one run of 16 sites at a time; lanes 0..15 hold the first flavour.

// even sites: t_e = kappa^2 A^-1 H psi  (DAG: kappa^2 A(-mu)^-1 H gamma_5 psi)
template <bool DAG>
__global__ void __launch_bounds__(FX_THREADS, FX_BLOCKS) k_fx_even(LatGeom g, FxSite st, const int4 *__restrict__ links,
                                                                   FxIn psi, FxOut out, const int *done,
                                                                   int nrun, FxBatch bt) {
    __shared__ FxShared sm;
    dependent_begin();
    if (done && *done) return;
    psi = fx_next(psi, blockIdx.y * bt.stride);
    out = fx_next(out, blockIdx.y * bt.stride);
    const int lane = threadIdx.x & 31, f = lane >> 4, s = threadIdx.x >> 5;
    const int r0 = (int)((long long)nrun * blockIdx.x / gridDim.x),
              r1 = (int)((long long)nrun * (blockIdx.x + 1) / gridDim.x);
    // A^-1 = [[1 - i kp g, kpp],[kpp, 1 + i kp g]] / det, g = gamma_5 eigenvalue; first flavour
    // o.re = a p.re + b p.im + c p'.re, o.im = a p.im - b p.re + c p'.im, b with the sign of g, of
    // the flavour and of mu
    const bool flip = (DAG != (f == 1)) != (s >= 2);
    const int2 b = flip ? make_int2(-st.inv_b.x, -st.inv_b.y) : st.inv_b;
    const int2 nb = make_int2(-b.x, -b.y);
    for (int run = r0; run < r1; run++) {
        const int hh = run * 16 + (lane & 15), h = min(hh, g.Vh - 1);
        long long v[3][2];
        const int em = hop_run<0, DAG>(g, links, psi.q + f * 12 * FX_RUN, psi.e, h, sm, v);
        const int L = norm_shift(v, sm);
        const bool zero = L == 64, nan = fx_is_nan(em);
        const int Ls = zero ? 0 : L;
        int ph[3][2], pl[3][2];
#pragma unroll
        for (int c = 0; c < 3; c++)
#pragma unroll
            for (int k = 0; k < 2; k++) norm_split(v[c][k], Ls, ph[c][k], pl[c][k]);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            int q[4];
#pragma unroll
            for (int k = 0; k < 2; k++) {
                const int oh = __shfl_xor_sync(0xffffffffu, ph[c][k], 16);
                const int ol = __shfl_xor_sync(0xffffffffu, pl[c][k], 16);
                long long x = 1ll << 27, y = 0;
                mac(st.inv_a, ph[c][k], pl[c][k], x, y);
                mac(k == 0 ? b : nb, ph[c][1 - k], pl[c][1 - k], x, y);
                mac(st.inv_c, oh, ol, x, y);
                fx_split(y + (x >> 28), q[2 * k], q[2 * k + 1]);
            }
            if (hh < g.Vh) out.q[fx_at(h, 24) + (f * 12 + s * 3 + c) * FX_RUN] = make_int4(q[0], q[1], q[2], q[3]);
        }
        if (hh < g.Vh && threadIdx.x < 16) out.e[h] = nan ? FX_NAN : zero ? FX_ZERO : em - Ls + 6 + st.inv_e;
    }
}

// odd sites: y = A psi - H t  (DAG: A(-mu) psi - gamma_5 H t), then the epilogue.
template <bool DAG, int EPI>
__global__ void __launch_bounds__(FX_THREADS, FX_BLOCKS) k_fx_odd(LatGeom g, FxSite st, const int4 *__restrict__ links,
                                                                  FxIn psi, FxIn te, FxOdd ea, int nrun, FxBatch bt) {
    __shared__ FxShared sm;
    __shared__ double red[40];
    dependent_begin();
    if (ea.done && *ea.done) return;
    psi = fx_next(psi, blockIdx.y * bt.stride);
    te = fx_next(te, blockIdx.y * bt.stride);
    if (EPI == FX_STORE) ea.out = fx_next(ea.out, blockIdx.y * bt.stride);
    const size_t off64 = blockIdx.y * bt.n64;
    const int lane = threadIdx.x & 31, f = lane >> 4, s = threadIdx.x >> 5, Vh = g.Vh;
    const double alpha = EPI == FX_MMS_R ? *ea.alpha : 0.0;
    double n1 = 0.0, n2 = 0.0;
    const int r0 = (int)((long long)nrun * blockIdx.x / gridDim.x),
              r1 = (int)((long long)nrun * (blockIdx.x + 1) / gridDim.x);
    // A = [[1 + i kp g, -kpp],[-kpp, 1 - i kp g]]: y.re = psi.re - b psi.im - kpp psi'.re,
    // y.im = psi.im + b psi.re - kpp psi'.im, b with the sign of g, of the flavour and of mu
    const bool flip = (DAG != (f == 1)) != (s >= 2);
    const int2 b = flip ? make_int2(-st.fwd_b.x, -st.fwd_b.y) : st.fwd_b;
    const int2 nb = make_int2(-b.x, -b.y);
    const bool plus = DAG && s >= 2;  // gamma_5 on the hop term
    for (int run = r0; run < r1; run++) {
        const int hh = run * 16 + (lane & 15), h = min(hh, Vh - 1);
        const bool in_range = hh < Vh;
        const int at = fx_at(h, 24) + (f * 12 + s * 3) * FX_RUN, ot = fx_at(h, 24) + ((1 - f) * 12 + s * 3) * FX_RUN;
        long long v[3][2];
        const int eh = hop_run<1, false>(g, links, te.q + f * 12 * FX_RUN, te.e, h, sm, v);
        const int ep = psi.e[h];
        const int ez = ep + st.fwd_e;
        int em = max(ez - 4, eh), es = FX_ZERO;
        if (EPI == FX_MMS_R) {
            es = ea.p.e[h] + ea.sig_e;
            em = max(em, es - 4);
        }
        const int sa = min(em - eh, 63), sz = min(em - (ez - 4), 63), ss = min(em - (es - 4), 63);
        long long pn_y = 0, pn_x = 0;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const int4 p = psi.q[at + c * FX_RUN];
            const int4 o = psi.q[ot + c * FX_RUN];
            int4 pp;
            if (EPI == FX_MMS_R) pp = ea.p.q[at + c * FX_RUN];
            const int ph[2] = {p.x, p.z}, pl[2] = {p.y, p.w};
            const int oh[2] = {o.x, o.z}, ol[2] = {o.y, o.w};
#pragma unroll
            for (int k = 0; k < 2; k++) {
                long long x = 1ll << 27, y = 0;
                mac(st.fwd_a, ph[k], pl[k], x, y);
                mac(k == 0 ? nb : b, ph[1 - k], pl[1 - k], x, y);
                mac(st.fwd_c, oh[k], ol[k], x, y);
                y += x >> 28;
                const long long hop = v[c][k] >> sa;
                long long w = ((y << 4) >> sz) + (plus ? hop : -hop);
                if (EPI == FX_MMS_R) {
                    long long x2 = 1ll << 27, y2 = 0;
                    mac(ea.sig, k == 0 ? pp.x : pp.z, k == 0 ? pp.y : pp.w, x2, y2);
                    w += ((y2 + (x2 >> 28)) << 4) >> ss;
                }
                v[c][k] = w;
                if (EPI == FX_STORE_NORMS) {
                    pn_y += (long long)ph[k] * ph[k];
                    pn_x += (long long)ph[k] * pl[k];
                }
            }
        }
        const bool nan = fx_is_nan(em);
        if (EPI == FX_STORE || EPI == FX_STORE_NORMS) {
            const int L = norm_shift(v, sm);
            const bool zero = L == 64;
            const int Ls = zero ? 0 : L;
            const int e_out = nan ? FX_NAN : zero ? FX_ZERO : em - Ls + 6;
            long long yn_y = 0, yn_x = 0;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                int4 w;
                norm_split(v[c][0], Ls, w.x, w.y);
                norm_split(v[c][1], Ls, w.z, w.w);
                if (in_range) ea.out.q[at + c * FX_RUN] = w;
                if (EPI == FX_STORE_NORMS) {
                    yn_y += (long long)w.x * w.x;
                    yn_x += (long long)w.x * w.y;
                    yn_y += (long long)w.z * w.z;
                    yn_x += (long long)w.z * w.w;
                }
            }
            if (in_range && threadIdx.x < 16) ea.out.e[h] = e_out;
            if (EPI == FX_STORE_NORMS && in_range) {
                // |v|^2 of the lane's words h 2^28 + l: (sum h h + sum h l / 2^27) 2^(2 e - 56)
                const FxScale s1 = fx_scale(e_out, e_out - 28), s2 = fx_scale(ep, ep - 28);
                n1 += fx_to_double(1, s1) * ((double)(yn_y + (yn_x >> 27)) * fx_to_double(1, s1));
                n2 += fx_to_double(1, s2) * ((double)(pn_y + (pn_x >> 27)) * fx_to_double(1, s2));
            }
        } else {
            const FxScale sc = fx_scale(em, em - 56);
            const double al = EPI == FX_MMS_R ? -alpha * sc.s1 : 0.0;
            double2 aux[3];  // loaded before the first store, which plain loads may not pass
            if (EPI == FX_F64_SHIFT || EPI == FX_RESID) {
#pragma unroll
                for (int c = 0; c < 3; c++) aux[c] = ea.aux64[off64 + (size_t)(f * 12 + s * 3 + c) * Vh + h];
            }
#pragma unroll
            for (int c = 0; c < 3; c++) {
                const size_t i = (size_t)(f * 12 + s * 3 + c) * Vh + h;
                const long long vr = v[c][0], vi = v[c][1];
                if (!in_range) continue;
                if (EPI == FX_F64) {
                    ea.out64[off64 + i] = make_double2(fx_to_double(vr, sc), fx_to_double(vi, sc));
                } else if (EPI == FX_F64_QHAT) {
                    // gamma_5 tau_1: the other flavour's slot, lower spins negated
                    const size_t j = (size_t)((1 - f) * 12 + s * 3 + c) * Vh + h;
                    const double sg = s < 2 ? 1.0 : -1.0;
                    ea.out64[off64 + j] = make_double2(sg * fx_to_double(vr, sc), sg * fx_to_double(vi, sc));
                } else if (EPI == FX_F64_SHIFT) {
                    const double2 a = aux[c];
                    ea.out64[off64 + i] = make_double2(fma(ea.sigma, a.x, fx_to_double(vr, sc)),
                                                       fma(ea.sigma, a.y, fx_to_double(vi, sc)));
                } else if (EPI == FX_RESID) {
                    const double2 a = aux[c], bv = ea.b64[i];
                    const double2 r1 = make_double2(bv.x - fma(ea.sigma, a.x, fx_to_double(vr, sc)),
                                                    bv.y - fma(ea.sigma, a.y, fx_to_double(vi, sc)));
                    ea.r[i] = r1;
                    n1 = fma(r1.x, r1.x, fma(r1.y, r1.y, n1));
                } else {  // FX_MMS_R: r' = r - alpha w
                    const double2 r0v = ea.r_in[i];
                    double wr = (double)vr, wi = (double)vi;
                    if (sc.split) {
                        wr *= sc.s2;
                        wi *= sc.s2;
                    }
                    const double2 r1 = make_double2(fma(al, wr, r0v.x), fma(al, wi, r0v.y));
                    ea.r[i] = r1;
                    n1 = fma(r1.x, r1.x, fma(r1.y, r1.y, n1));
                }
            }
            __syncthreads();  // the next run's parts overwrite this one's
        }
    }
    if (EPI == FX_STORE_NORMS) {
        double s1 = block_sum(n1, red);
        double s2 = block_sum(n2, red);
        if (threadIdx.x == 0) {
            ea.part_out[blockIdx.x] = s1;
            ea.part_out[gridDim.x + blockIdx.x] = s2;
        }
    } else if (EPI == FX_MMS_R || EPI == FX_RESID) {
        double s1 = block_sum(n1, red);
        if (threadIdx.x == 0) ea.part_out[blockIdx.x] = s1;
    }
}

// FP64 planes -> digits
__global__ void __launch_bounds__(128) k_fx_from_f64(int Vh, const double2 *in, FxOut out, FxBatch bt) {
    dependent_begin();
    in += blockIdx.y * bt.n64;
    out = fx_next(out, blockIdx.y * bt.stride);
    const int lane = threadIdx.x & 31, f = lane >> 4;
    const int gr = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int hh = gr * 16 + (lane & 15), h = min(hh, Vh - 1);
    double2 v[12];
#pragma unroll
    for (int c = 0; c < 12; c++) v[c] = in[(size_t)(f * 12 + c) * Vh + h];
    int4 q[12];
    int e;
    fx_from_doubles(v, q, e);
    if (hh >= Vh) return;
#pragma unroll
    for (int c = 0; c < 12; c++) out.q[fx_at(h, 24) + (f * 12 + c) * FX_RUN] = q[c];
    if (f == 0) out.e[h] = e;
}

// digits -> FP32 planes, scaled
__global__ void __launch_bounds__(256) k_fx_to_f32(int Vh, double a, FxIn in, float2 *__restrict__ out) {
    const int h = blockIdx.x * blockDim.x + threadIdx.x;
    if (h >= Vh) return;
    const size_t i = (size_t)blockIdx.y * Vh + h;
    const int e = in.e[h];
    const FxScale sc = fx_scale(e, e - 56);
    const int4 q = in.q[fx_at(h, 24) + (int)blockIdx.y * FX_RUN];
    out[i] = make_float2((float)(a * fx_to_double(fx_word(q.x, q.y), sc)),
                         (float)(a * fx_to_double(fx_word(q.z, q.w), sc)));
}

// p = r + beta p on digits (the base search direction of the multi-shift CG)
__global__ void __launch_bounds__(128) k_fx_pupdate(int Vh, const int *__restrict__ skip,
                                                    const double *__restrict__ beta_p,
                                                    const double2 *__restrict__ r, FxOut p) {
    if (*skip) return;
    const double beta = *beta_p;
    const int lane = threadIdx.x & 31, f = lane >> 4;
    const int gr = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
    const int hh = gr * 16 + (lane & 15), h = min(hh, Vh - 1);
    const int at = fx_at(h, 24) + f * 12 * FX_RUN;
    const int e0 = p.e[h];
    const FxScale sc = fx_scale(e0, e0 - 56);
    const double bs = beta * sc.s1;
    double2 v[12];
#pragma unroll
    for (int c = 0; c < 12; c++) {
        const size_t i = (size_t)(f * 12 + c) * Vh + h;
        const double2 rv = r[i];
        const int4 q = p.q[at + c * FX_RUN];
        double a = (double)fx_word(q.x, q.y), b = (double)fx_word(q.z, q.w);
        if (sc.split) {
            a *= sc.s2;
            b *= sc.s2;
        }
        v[c] = make_double2(fma(bs, a, rv.x), fma(bs, b, rv.y));
    }
    int4 q[12];
    int e;
    fx_from_doubles(v, q, e);
    if (hh >= Vh) return;
#pragma unroll
    for (int c = 0; c < 12; c++) p.q[at + c * FX_RUN] = q[c];
    if (f == 0) p.e[h] = e;
}

// canonical complex128 [4][T][X][Y][Z][3][3] -> digits [2 parity][4 mu] in runs of 16 sites, antiperiodic sign included
__global__ void k_fx_pack_links(Geom g, const double2 *__restrict__ canon, int4 *__restrict__ out) {
    const long V = 2L * g.Vh;
    const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;  // over 4 * V * 9
    if (i >= 4 * V * 9) return;
    const int k = (int)(i % 9);
    const long rest = i / 9;
    const long lex = rest % V;
    const int mu = (int)(rest / V);
    long r = lex;
    const int z = (int)(r % g.Z); r /= g.Z;
    const int y = (int)(r % g.Y); r /= g.Y;
    const int x = (int)(r % g.X);
    const int t = (int)(r / g.X);
    const int par = (t + x + y + z) & 1;
    const double sg = mu == 0 && t == g.T - 1 && g.apbc ? -1.0 : 1.0;
    const double2 u = canon[i];
    int4 w;
    fx_split(llrint(sg * u.x * 72057594037927936.0), w.x, w.y);  // 2^56
    fx_split(llrint(sg * u.y * 72057594037927936.0), w.z, w.w);
    const size_t Vs = (g.Vh + 15) & ~15;
    out[((size_t)par * 4 + mu) * 9 * Vs + fx_at((int)(lex >> 1), 9) + k * FX_RUN] = w;
}

// digits of x 2^-e, |x 2^-e| <= 1 (host)
int2 digits(double x, int e) {
    const long long q = llrint(ldexp(x, 56 - e));
    const long long t = q + (1ll << 27);
    return make_int2((int)(t >> 28), (int)(t & 0x0fffffff) - (1 << 27));
}
int exponent_of(double x) {  // smallest e with |x| <= 2^e
    int e = 0;
    const double m = frexp(x, &e);
    return fabs(m) == 0.5 ? e - 1 : e;
}

}  // namespace

FxSite fx_site(const SiteTerm &st) {
    FxSite r;
    const double a = st.kappa2 * st.inv_det, b = a * st.kp, c = a * st.kpp;
    r.inv_e = exponent_of(fabs(a) + fabs(b) + fabs(c));
    r.inv_a = digits(a, r.inv_e);
    r.inv_b = digits(b, r.inv_e);
    r.inv_c = digits(c, r.inv_e);
    r.fwd_e = exponent_of(1.0 + fabs(st.kp) + fabs(st.kpp));
    r.fwd_a = digits(1.0, r.fwd_e);
    r.fwd_b = digits(st.kp, r.fwd_e);
    r.fwd_c = digits(-st.kpp, r.fwd_e);
    return r;
}

namespace {
struct FxGrid {
    int blocks, runs, cap;
};
// As many blocks as fit on the chip at once (the reductions then need few partials), each with a
// contiguous stretch of runs of about the same length.  Per SM 4, 5, 6: 3.53, 3.43, 3.76 ms for Qhat^2 at
// 32^3x64 (6 spills).
FxGrid fx_grid(int Vh) {
    static int sms[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!sms[dev]) {
        int n = 0;
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        sms[dev] = n > 0 ? n : 152;
    }
    const int runs = (Vh + 15) / 16, cap = sms[dev] * FX_BLOCKS;
    return FxGrid{runs < cap ? runs : cap, runs, cap};
}
}  // namespace

int fx_blocks(const Geom &g) { return fx_grid(g.Vh).blocks; }

int fx_batch(const Geom &g, int nrhs) {
    const FxGrid r = fx_grid(g.Vh);
    const int most = 1 + 2 * r.cap / r.runs;
    return nrhs < most ? nrhs : most;
}

void launch_fx_from_f64(const Geom &g, const double2 *in, FxOut out, cudaStream_t s, const FxBatch &bt) {
    const int groups = (g.Vh + 15) / 16;
    launch_dependent(k_fx_from_f64, dim3((groups + 3) / 4, bt.nrhs), 128, s, g.Vh, in, out, bt);
}

void launch_fx_to_f32(const Geom &g, double a, FxIn in, float2 *out, cudaStream_t s) {
    k_fx_to_f32<<<dim3((g.Vh + 255) / 256, NCOMP), 256, 0, s>>>(g.Vh, a, in, out);
}

void launch_fx_pupdate(const Geom &g, const int *skip, const double *beta, const double2 *r, FxOut p,
                       cudaStream_t s) {
    const int groups = (g.Vh + 15) / 16;
    k_fx_pupdate<<<(groups + 3) / 4, 128, 0, s>>>(g.Vh, skip, beta, r, p);
}

void launch_fx_pack_links(const Geom &g, const double2 *canon, int4 *out, cudaStream_t s) {
    const long n = 4L * 2 * g.Vh * 9;
    k_fx_pack_links<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(g, canon, out);
}

void launch_fx_even(const Geom &g, const FxSite &st, const int4 *links, FxIn psi, FxOut out, bool dag,
                    const int *done, cudaStream_t s, const FxBatch &bt) {
    const FxGrid gr = fx_grid(g.Vh);
    const LatGeom fg = lat_geom(g);
    if (dag)
        launch_dependent(k_fx_even<true>, dim3(gr.blocks, bt.nrhs), FX_THREADS, s, fg, st, links, psi, out, done, gr.runs, bt);
    else
        launch_dependent(k_fx_even<false>, dim3(gr.blocks, bt.nrhs), FX_THREADS, s, fg, st, links, psi, out, done, gr.runs, bt);
}

void launch_fx_odd(const Geom &g, const FxSite &st, const int4 *links, FxIn psi, FxIn te, bool dag, FxEpi epi,
                   FxOdd ea, cudaStream_t s, const FxBatch &bt) {
    const FxGrid gr = fx_grid(g.Vh);
    const LatGeom fg = lat_geom(g);
    if (epi == FX_MMS_R) {
        ea.sig_e = exponent_of(ea.sigma);
        ea.sig = digits(ea.sigma, ea.sig_e);
    }
#define TMND_FX(D, E) launch_dependent(k_fx_odd<D, E>, dim3(gr.blocks, bt.nrhs), FX_THREADS, s, fg, st, links, psi, te, ea, gr.runs, bt)
    switch (epi) {
        case FX_STORE: dag ? TMND_FX(true, FX_STORE) : TMND_FX(false, FX_STORE); break;
        case FX_STORE_NORMS: TMND_FX(false, FX_STORE_NORMS); break;
        case FX_F64: dag ? TMND_FX(true, FX_F64) : TMND_FX(false, FX_F64); break;
        case FX_F64_QHAT: TMND_FX(false, FX_F64_QHAT); break;
        case FX_F64_SHIFT: TMND_FX(true, FX_F64_SHIFT); break;
        case FX_RESID: TMND_FX(true, FX_RESID); break;
        case FX_MMS_R: TMND_FX(true, FX_MMS_R); break;
    }
#undef TMND_FX
}
