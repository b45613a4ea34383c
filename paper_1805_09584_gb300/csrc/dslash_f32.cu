// FP32 hopping kernels: the even-odd reduced ND twisted-mass operator on FP32 planes with 18-real FP32
// links, accurate to ~1e-7 (the inner residuals of the defect correction, and single-precision callers of
// tm_nd_apply), and the full-lattice operator of the multigrid.
//
//   even kernel:  t_e = kappa^2 A^-1 H_eo psi_o
//   odd  kernel:  y_o = A psi_o - H_oe t_e                 => y = Mhat psi  (Sec. 2 even-odd reduction)
//   dagger:       Mhat^+ = gamma_5 Mhat(-mu_bar) gamma_5     (A and gamma_5 commute; H is gamma_5-hermitian)
//                 even: kappa^2 A(-mu)^-1 H_eo gamma_5 psi_o
//                 odd : A(-mu) psi_o - gamma_5 H_oe t_e
//   full lattice: D' x = A x - kappa H x + i s gamma_5 tau_1 x on odd sites
//
// The hop and its spin projection are those of hop_fx.cu.  A thread owns one site and one flavour (lanes
// 0..15 of a warp the first, 16..31 the second, of the same 16 sites), so that 24 accumulators and one link
// are live: 128 registers and 16 warps per SM, where one thread for both flavours took 255 (Qhat^2 at
// 24^3x48: 488 -> 319 us against 216 us of HBM time; 5 and 6 blocks per SM spill: 435, 447 us).
#include "lattice.cuh"
#include "launch.cuh"

namespace {

constexpr int F32_THREADS = 128, F32_BLOCKS = 4;

// (B_mu v) for the lower two spins, v[2][3]
template <int MU>
__device__ __forceinline__ float2 Bmul(const float2 v[2][3], int s, int c) {
    if (MU == 0) return cneg(v[s][c]);
    if (MU == 1) return cmulmi(v[1 - s][c]);                 // -i sigma_1
    if (MU == 2) return s == 0 ? cneg(v[1][c]) : v[0][c];    // -i sigma_2 = [[0,-1],[1,0]]
    return s == 0 ? cmulmi(v[0][c]) : cmuli(v[1][c]);        // -i sigma_3 = diag(-i, i)
}

// (B_mu^+ v)
template <int MU>
__device__ __forceinline__ float2 Bdag(const float2 v[2][3], int s, int c) {
    if (MU == 0) return cneg(v[s][c]);
    if (MU == 1) return cmuli(v[1 - s][c]);                  // i sigma_1
    if (MU == 2) return s == 0 ? v[1][c] : cneg(v[0][c]);    // i sigma_2 = [[0,1],[-1,0]]
    return s == 0 ? cmuli(v[0][c]) : cmulmi(v[1][c]);        // i sigma_3 = diag(i, -i)
}

// Accumulate the hop from the neighbour at `in` (its first plane) in direction MU, DIR (+1 forward with
// U_mu(x), -1 backward with U_mu(x-mu)^+) into acc[spin][colour]; sg = -1 across the antiperiodic boundary.
// G5IN: the input field is gamma_5 psi (lower spins negated).
template <int MU, int DIR, bool G5IN>
__device__ __forceinline__ void hop_dir(const float2 *in, const float2 *__restrict__ U, int Vh, float sg,
                                        float2 acc[4][3]) {
    // sign of the B psi_lo term in chi: forward -, backward +; gamma_5 on input flips it
    constexpr bool plus = (DIR < 0) != G5IN;
    float2 up[2][3], lo[2][3];
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            up[s][c] = in[(s * 3 + c) * Vh];
            lo[s][c] = in[((s + 2) * 3 + c) * Vh];
        }
    float2 chi[2][3];
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 b = Bmul<MU>(lo, s, c);
            chi[s][c] = plus ? cadd(up[s][c], b) : csub(up[s][c], b);
        }
    float2 v[2][3];
#pragma unroll
    for (int i = 0; i < 3; i++) {
        float2 u[3];
#pragma unroll
        for (int j = 0; j < 3; j++) u[j] = __ldg(&U[(DIR > 0 ? i * 3 + j : j * 3 + i) * Vh]);
#pragma unroll
        for (int s = 0; s < 2; s++)
            v[s][i] = DIR > 0 ? cfma(u[2], chi[s][2], cfma(u[1], chi[s][1], cmul(u[0], chi[s][0])))
                              : cfma_conj(u[2], chi[s][2], cfma_conj(u[1], chi[s][1], cmul_conj(u[0], chi[s][0])));
    }
#pragma unroll
    for (int s = 0; s < 2; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 b = Bdag<MU>(v, s, c);
            float2 &a = acc[s][c], &l = acc[s + 2][c];
            const float f = MU == 0 ? sg : 1.0f, fl = DIR > 0 ? -f : f;
            a = make_float2(fmaf(f, v[s][c].x, a.x), fmaf(f, v[s][c].y, a.y));
            l = make_float2(fmaf(fl, b.x, l.x), fmaf(fl, b.y, l.y));
        }
}

// H applied at output site h of parity P to one flavour; in: that flavour's planes on parity 1 - P.
template <int P, bool G5IN>
__device__ __forceinline__ void hop_all(const LatGeom &g, int apbc, const float2 *__restrict__ links,
                                        const float2 *in, int h, float2 acc[4][3]) {
    const int Vh = g.Vh;
    const float2 *Lp = links + (size_t)P * 4 * 9 * Vh;        // links based at parity P sites
    const float2 *Lq = links + (size_t)(1 - P) * 4 * 9 * Vh;  // links based at parity 1-P sites
#pragma unroll
    for (int s = 0; s < 4; s++)
#pragma unroll
        for (int c = 0; c < 3; c++) acc[s][c] = make_float2(0.f, 0.f);
    const int r = fdiv(h, g.dZh), zh = h - r * g.Zh, q = fdiv(r, g.dY), y = r - q * g.Y;
    const int t = fdiv(q, g.dX), x = q - t * g.X;
    const bool odd = (P + t + x + y) & 1;  // z = 2 zh + odd
    int hf, hb;
    hf = t + 1 == g.T ? h - (g.T - 1) * g.st : h + g.st;
    hb = t == 0 ? h + (g.T - 1) * g.st : h - g.st;
    hop_dir<0, +1, G5IN>(in + hf, Lp + h, Vh, apbc && t + 1 == g.T ? -1.0f : 1.0f, acc);
    hop_dir<0, -1, G5IN>(in + hb, Lq + hb, Vh, apbc && t == 0 ? -1.0f : 1.0f, acc);
    hf = x + 1 == g.X ? h - (g.X - 1) * g.sx : h + g.sx;
    hb = x == 0 ? h + (g.X - 1) * g.sx : h - g.sx;
    hop_dir<1, +1, G5IN>(in + hf, Lp + 9 * (size_t)Vh + h, Vh, 1.0f, acc);
    hop_dir<1, -1, G5IN>(in + hb, Lq + 9 * (size_t)Vh + hb, Vh, 1.0f, acc);
    hf = y + 1 == g.Y ? h - (g.Y - 1) * g.Zh : h + g.Zh;
    hb = y == 0 ? h + (g.Y - 1) * g.Zh : h - g.Zh;
    hop_dir<2, +1, G5IN>(in + hf, Lp + 18 * (size_t)Vh + h, Vh, 1.0f, acc);
    hop_dir<2, -1, G5IN>(in + hb, Lq + 18 * (size_t)Vh + hb, Vh, 1.0f, acc);
    hf = !odd ? h : zh + 1 == g.Zh ? h - (g.Zh - 1) : h + 1;
    hb = odd ? h : zh == 0 ? h + (g.Zh - 1) : h - 1;
    hop_dir<3, +1, G5IN>(in + hf, Lp + 27 * (size_t)Vh + h, Vh, 1.0f, acc);
    hop_dir<3, -1, G5IN>(in + hb, Lq + 27 * (size_t)Vh + hb, Vh, 1.0f, acc);
}

struct SiteTerm32 {
    float a, b, e;   // kappa^2 A^-1 = a (1 - i kp g tau_3 + kpp tau_1), b = a kp, e = a kpp
    float kp, kpp;
};
SiteTerm32 site32(const SiteTerm &st, bool dag) {
    SiteTerm32 r;
    r.a = (float)(st.kappa2 * st.inv_det);
    r.kp = (float)(dag ? -st.kp : st.kp);
    r.kpp = (float)st.kpp;
    r.b = r.a * r.kp;
    r.e = (float)(st.kappa2 * st.inv_det * st.kpp);
    return r;
}

// even sites: t_e = kappa^2 A^-1 H psi  (DAG: kappa^2 A(-mu)^-1 H gamma_5 psi); right-hand side blockIdx.y
template <bool DAG>
__global__ void __launch_bounds__(F32_THREADS, F32_BLOCKS) k_even_f32(LatGeom g, int apbc, SiteTerm32 st,
                                                                     const float2 *__restrict__ links,
                                                                     const float2 *psi,
                                                                     float2 *__restrict__ out) {
    dependent_begin();
    const int lane = threadIdx.x & 31, f = lane >> 4, Vh = g.Vh;
    const int hh = (blockIdx.x * (F32_THREADS / 32) + (threadIdx.x >> 5)) * 16 + (lane & 15), h = min(hh, Vh - 1);
    const size_t off = (size_t)blockIdx.y * NCOMP * Vh + (size_t)f * 12 * Vh;
    float2 acc[4][3];
    hop_all<0, DAG>(g, apbc, links, psi + off, h, acc);
    float2 *o = out + off + h;
#pragma unroll
    for (int s = 0; s < 4; s++) {
        const float b = (f == 0) == (s < 2) ? st.b : -st.b;  // sign of gamma_5 and of the flavour
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 p = acc[s][c];
            const float qx = __shfl_xor_sync(0xffffffffu, p.x, 16), qy = __shfl_xor_sync(0xffffffffu, p.y, 16);
            const float2 r = make_float2(fmaf(st.a, p.x, fmaf(b, p.y, st.e * qx)), fmaf(st.a, p.y, fmaf(-b, p.x, st.e * qy)));
            if (hh < Vh) o[(s * 3 + c) * Vh] = r;
        }
    }
}

// odd sites: y = A psi - H t  (DAG: A(-mu) psi - gamma_5 H t); EPI_SHIFT adds sigma aux
template <bool DAG, int EPI>
__global__ void __launch_bounds__(F32_THREADS, F32_BLOCKS) k_odd_f32(LatGeom g, int apbc, SiteTerm32 st,
                                                                    const float2 *__restrict__ links,
                                                                    const float2 *psi,
                                                                    const float2 *te,
                                                                    float2 *__restrict__ out, HopEpiArgsF ea) {
    dependent_begin();
    const int lane = threadIdx.x & 31, f = lane >> 4, Vh = g.Vh;
    const int hh = (blockIdx.x * (F32_THREADS / 32) + (threadIdx.x >> 5)) * 16 + (lane & 15), h = min(hh, Vh - 1);
    const size_t off = (size_t)blockIdx.y * NCOMP * Vh + (size_t)f * 12 * Vh;
    float2 acc[4][3];
    hop_all<1, false>(g, apbc, links, te + off, h, acc);
    if (hh >= Vh) return;
    const float sigma = EPI == EPI_SHIFT ? ea.sigma[ea.per_rhs ? blockIdx.y : 0] : 0.0f;
    const float2 *own = psi + off + h, *oth = psi + (size_t)blockIdx.y * NCOMP * Vh + (size_t)(1 - f) * 12 * Vh + h;
    float2 *o = out + off + h;
    float2 po[12], qo[12], ao[12];  // all loads before the first store, which plain loads may not pass
#pragma unroll
    for (int k = 0; k < 12; k++) {
        po[k] = own[k * Vh];
        qo[k] = oth[k * Vh];
        if (EPI == EPI_SHIFT) ao[k] = ea.aux[off + h + (size_t)k * Vh];
    }
#pragma unroll
    for (int s = 0; s < 4; s++) {
        const float b = (f == 0) == (s < 2) ? st.kp : -st.kp;
        // DAG: gamma_5 on the hop term flips the sign of the lower spins
        const bool hopneg = DAG && s >= 2;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 p = po[s * 3 + c], q = qo[s * 3 + c];
            const float2 hp = hopneg ? cneg(acc[s][c]) : acc[s][c];
            // A = [[1 + i kp g, -kpp],[-kpp, 1 - i kp g]]
            float2 y = make_float2(fmaf(-b, p.y, fmaf(-st.kpp, q.x, p.x - hp.x)), fmaf(b, p.x, fmaf(-st.kpp, q.y, p.y - hp.y)));
            if (EPI == EPI_SHIFT) {
                const float2 a = ao[s * 3 + c];
                y = make_float2(fmaf(sigma, a.x, y.x), fmaf(sigma, a.y, y.y));
            }
            o[(s * 3 + c) * Vh] = y;
        }
    }
}

// Full lattice, vectors [parity][12 NF][V/2], output parity blockIdx.y: y = A x - kappa H x, on odd sites
// + i s gamma_5 tau_1 x.  NF = 1: one flavour, D_TM(+mu) (kpp and s ignored), 32 sites per warp.
template <int NF, int P>
__device__ __forceinline__ void dnd_sites(const LatGeom &g, int apbc, float kappa, float kp, float kpp, float so,
                                          const float2 *__restrict__ links, const float2 *in,
                                          float2 *__restrict__ out) {
    const int lane = threadIdx.x & 31, f = NF == 2 ? lane >> 4 : 0, Vh = g.Vh;
    constexpr int SITES = NF == 2 ? 16 : 32;
    const int h = (blockIdx.x * (F32_THREADS / 32) + (threadIdx.x >> 5)) * SITES + (lane & (SITES - 1));
    if (h >= Vh) return;
    const size_t n = (size_t)NF * 12 * Vh;
    float2 acc[4][3];
    hop_all<P, false>(g, apbc, links, in + (1 - P) * n + (size_t)f * 12 * Vh, h, acc);
    const float2 *own = in + P * n + (size_t)f * 12 * Vh + h, *oth = in + P * n + (size_t)(NF - 1 - f) * 12 * Vh + h;
    float2 *o = out + P * n + (size_t)f * 12 * Vh + h;
    float2 po[12], qo[12];
#pragma unroll
    for (int k = 0; k < 12; k++) {
        po[k] = own[k * Vh];
        if (NF == 2) qo[k] = oth[k * Vh];
    }
#pragma unroll
    for (int s = 0; s < 4; s++) {
        const float g5 = s < 2 ? 1.0f : -1.0f;
        const float b = f == 0 ? kp * g5 : -kp * g5, e = P == 1 ? so * g5 : 0.0f;
#pragma unroll
        for (int c = 0; c < 3; c++) {
            const float2 p = po[s * 3 + c];
            float2 y = make_float2(fmaf(-b, p.y, fmaf(-kappa, acc[s][c].x, p.x)), fmaf(b, p.x, fmaf(-kappa, acc[s][c].y, p.y)));
            if (NF == 2) {
                const float2 q = qo[s * 3 + c];
                y = make_float2(fmaf(-kpp, q.x, fmaf(-e, q.y, y.x)), fmaf(-kpp, q.y, fmaf(e, q.x, y.y)));
            }
            o[(s * 3 + c) * Vh] = y;
        }
    }
}
template <int NF>
__global__ void __launch_bounds__(F32_THREADS, F32_BLOCKS) k_dnd(LatGeom g, int apbc, float kappa, float kp, float kpp,
                                                                float so, const float2 *__restrict__ links,
                                                                const float2 *in, float2 *__restrict__ out) {
    dependent_begin();
    if (blockIdx.y == 0) dnd_sites<NF, 0>(g, apbc, kappa, kp, kpp, so, links, in, out);
    else dnd_sites<NF, 1>(g, apbc, kappa, kp, kpp, so, links, in, out);
}

int blocks_of(int Vh, int sites_per_block) { return (Vh + sites_per_block - 1) / sites_per_block; }

}  // namespace

void launch_hop_even_f32(const Geom &g, const SiteTerm &st, const float2 *links, const float2 *psi_o, float2 *t_e,
                         bool dag, int nrhs, cudaStream_t s) {
    const dim3 grid(blocks_of(g.Vh, F32_THREADS / 2), nrhs);
    const SiteTerm32 t = site32(st, dag);
    if (dag)
        launch_dependent(k_even_f32<true>, grid, F32_THREADS, s, lat_geom(g), g.apbc, t, links, psi_o, t_e);
    else
        launch_dependent(k_even_f32<false>, grid, F32_THREADS, s, lat_geom(g), g.apbc, t, links, psi_o, t_e);
}

void launch_hop_odd_f32(const Geom &g, const SiteTerm &st, const float2 *links, const float2 *psi_o,
                        const float2 *t_e, float2 *y_o, bool dag, HopEpi epi, const HopEpiArgsF &ea, int nrhs,
                        cudaStream_t s) {
    const dim3 grid(blocks_of(g.Vh, F32_THREADS / 2), nrhs);
    const SiteTerm32 t = site32(st, dag);
#define TMND_ODD32(D, E) launch_dependent(k_odd_f32<D, E>, grid, F32_THREADS, s, lat_geom(g), g.apbc, t, links, psi_o, t_e, y_o, ea)
    if (epi == EPI_STORE) {
        dag ? TMND_ODD32(true, EPI_STORE) : TMND_ODD32(false, EPI_STORE);
    } else {
        TMND_ODD32(true, EPI_SHIFT);  // of Qhat^2 + sigma only
    }
#undef TMND_ODD32
}

void launch_dnd_full(const Geom &g, double kappa, float kp, float kpp, float s_odd, const float2 *links,
                     const float2 *in, float2 *out, int nf, cudaStream_t s) {
    if (nf == 2)
        launch_dependent(k_dnd<2>, dim3(blocks_of(g.Vh, F32_THREADS / 2), 2), F32_THREADS, s, lat_geom(g), g.apbc, (float)kappa, kp,
                                                                                  kpp, s_odd, links, in, out);
    else
        launch_dependent(k_dnd<1>, dim3(blocks_of(g.Vh, F32_THREADS), 2), F32_THREADS, s, lat_geom(g), g.apbc, (float)kappa, kp, kpp,
                                                                              s_odd, links, in, out);
}
