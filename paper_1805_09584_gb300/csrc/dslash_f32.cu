// FP32 hopping kernels for the even-odd reduced ND twisted-mass operator: FP32 planes,
// 18-real FP32 links, accurate to ~1e-7 (the inner residuals of the defect correction,
// and single-precision callers of tm_nd_apply).
//
//   even kernel:  t_e = kappa^2 A^-1 H_eo psi_o
//   odd  kernel:  y_o = A psi_o - H_oe t_e                 => y = Mhat psi  (Sec. 2 even-odd reduction)
//   dagger:       Mhat^+ = gamma_5 Mhat(-mu_bar) gamma_5     (A and gamma_5 commute; H is gamma_5-hermitian)
//                 even: kappa^2 A(-mu)^-1 H_eo gamma_5 psi_o
//                 odd : A(-mu) psi_o - gamma_5 H_oe t_e
//
// The hop and its spin projection are those of hop_fx.cu.  One thread owns one output site and both
// flavours, which share the eight links.
#include "tmnd_internal.cuh"

namespace {

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

// Accumulate the hop from neighbour hn in direction MU, DIR (+1 forward
// with U_mu(x), -1 backward with U_mu(x-mu)^+) into acc[flavour][spin][colour].
// G5IN: the input field is gamma_5 psi (lower spins negated).
template <int MU, int DIR, bool G5IN, bool FIRST = false>
__device__ __forceinline__ void hop_dir(const float2 *__restrict__ in, int Vh, int hn, const float2 *__restrict__ U, int hl,
                                        unsigned long long smask, float2 acc[2][4][3]) {
    float2 u[3][3];
#pragma unroll
    for (int i = 0; i < 3; i++)
#pragma unroll
        for (int j = 0; j < 3; j++) u[i][j] = __ldg(&U[(i * 3 + j) * Vh + hl]);
    // sign of the B psi_lo term in chi: forward -, backward +; gamma_5 on input flips it
    constexpr bool plus = (DIR < 0) != G5IN;
#pragma unroll
    for (int f = 0; f < 2; f++) {
        float2 up[2][3], lo[2][3];
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                up[s][c] = __ldg(&in[(f * 12 + s * 3 + c) * Vh + hn]);
                lo[s][c] = __ldg(&in[(f * 12 + (s + 2) * 3 + c) * Vh + hn]);
            }
        float2 chi[2][3];
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                float2 b = Bmul<MU>(lo, s, c);
                chi[s][c] = cflip(plus ? cadd(up[s][c], b) : csub(up[s][c], b), smask);
            }
        float2 v[2][3];
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int i = 0; i < 3; i++) {
                if (DIR > 0) {
                    float2 t = cmul(u[i][0], chi[s][0]);
                    t = cfma(u[i][1], chi[s][1], t);
                    v[s][i] = cfma(u[i][2], chi[s][2], t);
                } else {
                    float2 t = cmul_conj(u[0][i], chi[s][0]);
                    t = cfma_conj(u[1][i], chi[s][1], t);
                    v[s][i] = cfma_conj(u[2][i], chi[s][2], t);
                }
            }
#pragma unroll
        for (int s = 0; s < 2; s++)
#pragma unroll
            for (int c = 0; c < 3; c++) {
                float2 b = Bdag<MU>(v, s, c);
                if (FIRST) {  // the first direction initialises the accumulator
                    acc[f][s][c] = v[s][c];
                    acc[f][s + 2][c] = (DIR > 0) ? cneg(b) : b;
                } else {
                    acc[f][s][c] = cadd(acc[f][s][c], v[s][c]);
                    acc[f][s + 2][c] = (DIR > 0) ? csub(acc[f][s + 2][c], b) : cadd(acc[f][s + 2][c], b);
                }
            }
    }
}

// H applied at output site of parity P, half-index h; in = field on parity 1-P.
template <int P, bool G5IN>
__device__ __forceinline__ void hop_all(const Geom &g, const float2 *__restrict__ links, const float2 *__restrict__ in, int h,
                                        float2 acc[2][4][3]) {
    const int Vh = g.Vh;
    int zh = h % g.Zh;
    int r = h / g.Zh;
    int y = r % g.Y;
    r /= g.Y;
    int x = r % g.X;
    int t = r / g.X;
    int z = 2 * zh + ((P + t + x + y) & 1);
    const float2 *Lp = links + (size_t)P * 4 * 9 * Vh;         // links based at parity P sites
    const float2 *Lq = links + (size_t)(1 - P) * 4 * 9 * Vh;   // links based at parity 1-P sites
    const unsigned long long NEG = 0x8000000000000000ull;
    auto idx = [&](int tt, int xx, int yy, int zz) { return ((tt * g.X + xx) * g.Y + yy) * g.Zh + (zz >> 1); };

    // mu = 0 (time), with the antiperiodic sign on boundary-crossing hops
    {
        int tf = (t + 1 == g.T) ? 0 : t + 1;
        int tb = (t == 0) ? g.T - 1 : t - 1;
        unsigned long long mf = (g.apbc && t + 1 == g.T) ? NEG : 0ull;
        unsigned long long mb = (g.apbc && t == 0) ? NEG : 0ull;
        int hf = idx(tf, x, y, z), hb = idx(tb, x, y, z);
        hop_dir<0, +1, G5IN, true>(in, Vh, hf, Lp + 0 * 9 * (size_t)Vh, h, mf, acc);
        hop_dir<0, -1, G5IN>(in, Vh, hb, Lq + 0 * 9 * (size_t)Vh, hb, mb, acc);
    }
    {
        int xf = (x + 1 == g.X) ? 0 : x + 1;
        int xb = (x == 0) ? g.X - 1 : x - 1;
        int hf = idx(t, xf, y, z), hb = idx(t, xb, y, z);
        hop_dir<1, +1, G5IN>(in, Vh, hf, Lp + 1 * 9 * (size_t)Vh, h, 0ull, acc);
        hop_dir<1, -1, G5IN>(in, Vh, hb, Lq + 1 * 9 * (size_t)Vh, hb, 0ull, acc);
    }
    {
        int yf = (y + 1 == g.Y) ? 0 : y + 1;
        int yb = (y == 0) ? g.Y - 1 : y - 1;
        int hf = idx(t, x, yf, z), hb = idx(t, x, yb, z);
        hop_dir<2, +1, G5IN>(in, Vh, hf, Lp + 2 * 9 * (size_t)Vh, h, 0ull, acc);
        hop_dir<2, -1, G5IN>(in, Vh, hb, Lq + 2 * 9 * (size_t)Vh, hb, 0ull, acc);
    }
    {
        int zf = (z + 1 == g.Z) ? 0 : z + 1;
        int zb = (z == 0) ? g.Z - 1 : z - 1;
        int hf = idx(t, x, y, zf), hb = idx(t, x, y, zb);
        hop_dir<3, +1, G5IN>(in, Vh, hf, Lp + 3 * 9 * (size_t)Vh, h, 0ull, acc);
        hop_dir<3, -1, G5IN>(in, Vh, hb, Lq + 3 * 9 * (size_t)Vh, hb, 0ull, acc);
    }
}

// even sites: t_e = kappa^2 A^-1 H psi  (DAG: kappa^2 A(-mu)^-1 H gamma_5 psi)
template <bool DAG>
__global__ void __launch_bounds__(HOP_THREADS) k_hop_even(Geom g, SiteTerm st, const float2 *__restrict__ links,
                                                         const float2 *__restrict__ psi, float2 *__restrict__ out, int chunk) {
    const int h_end = min(g.Vh, (blockIdx.x + 1) * chunk);
    for (int h = blockIdx.x * chunk + threadIdx.x; h < h_end; h += blockDim.x) {
    float2 acc[2][4][3];
    hop_all<0, DAG>(g, links, psi, h, acc);
    const float a = (float)(st.kappa2 * st.inv_det);
    const float e = (float)(st.kappa2 * st.inv_det * st.kpp);
    const int Vh = g.Vh;
#pragma unroll
    for (int s = 0; s < 4; s++) {
        // A^-1 = [[1 - i kp g, kpp],[kpp, 1 + i kp g]] / det, g = gamma_5 eigenvalue
        const float b = a * (float)(DAG ? -st.kp : st.kp) * (s < 2 ? (float)1 : (float)-1);
#pragma unroll
        for (int c = 0; c < 3; c++) {
            float2 p0 = acc[0][s][c], p1 = acc[1][s][c];
            float2 o0, o1;
            o0.x = fma(a, p0.x, fma(b, p0.y, e * p1.x));
            o0.y = fma(a, p0.y, fma(-b, p0.x, e * p1.y));
            o1.x = fma(a, p1.x, fma(-b, p1.y, e * p0.x));
            o1.y = fma(a, p1.y, fma(b, p1.x, e * p0.y));
            out[(0 * 12 + s * 3 + c) * Vh + h] = o0;
            out[(1 * 12 + s * 3 + c) * Vh + h] = o1;
        }
    }
    }
}

// odd sites: y = A psi - H t  (DAG: A(-mu) psi - gamma_5 H t), then the epilogue.
template <bool DAG, int EPI>
__global__ void __launch_bounds__(HOP_THREADS) k_hop_odd(Geom g, SiteTerm st, const float2 *__restrict__ links,
                                                        const float2 *__restrict__ psi, const float2 *__restrict__ te,
                                                        float2 *__restrict__ out, HopEpiArgsF ea, int chunk) {
    const int Vh = g.Vh;
    const int h_end = min(Vh, (int)(blockIdx.x + 1) * chunk);
    for (int h = blockIdx.x * chunk + threadIdx.x; h < h_end; h += blockDim.x) {
        float2 acc[2][4][3];
        hop_all<1, false>(g, links, te, h, acc);
        const float kp = (float)(DAG ? -st.kp : st.kp);
        const float kpp = (float)st.kpp;
        const float sg = (float)ea.sigma;
#pragma unroll
        for (int s = 0; s < 4; s++) {
            const float b = kp * (s < 2 ? (float)1 : (float)-1);
            // DAG: gamma_5 on the hop term flips the sign of the lower spins
            const bool hopneg = DAG && s >= 2;
#pragma unroll
            for (int c = 0; c < 3; c++) {
                float2 p0 = __ldg(&psi[(0 * 12 + s * 3 + c) * Vh + h]);
                float2 p1 = __ldg(&psi[(1 * 12 + s * 3 + c) * Vh + h]);
                float2 h0 = acc[0][s][c], h1 = acc[1][s][c];
                if (hopneg) { h0 = cneg(h0); h1 = cneg(h1); }
                // A = [[1 + i kp g, -kpp],[-kpp, 1 - i kp g]]
                float2 y0, y1;
                y0.x = fma(-b, p0.y, fma(-kpp, p1.x, p0.x - h0.x));
                y0.y = fma(b, p0.x, fma(-kpp, p1.y, p0.y - h0.y));
                y1.x = fma(b, p1.y, fma(-kpp, p0.x, p1.x - h1.x));
                y1.y = fma(-b, p1.x, fma(-kpp, p0.y, p1.y - h1.y));
                const int i0 = (0 * 12 + s * 3 + c) * Vh + h, i1 = (1 * 12 + s * 3 + c) * Vh + h;
                if (EPI == EPI_STORE) {
                    out[i0] = y0;
                    out[i1] = y1;
                } else {  // EPI_SHIFT
                    float2 a0 = __ldg(&ea.aux[i0]), a1 = __ldg(&ea.aux[i1]);
                    out[i0] = make_float2(fmaf(sg, a0.x, y0.x), fmaf(sg, a0.y, y0.y));
                    out[i1] = make_float2(fmaf(sg, a1.x, y1.x), fmaf(sg, a1.y, y1.y));
                }
            }
        }
    }
}

}  // namespace

// Persistent, balanced grid: every SM gets the same number of resident blocks and every block a
// contiguous chunk of about the same number of sites.
static int hop_blocks_f32(const Geom &g) {
    static int cached[64] = {0};
    int dev = 0;
    cudaGetDevice(&dev);
    if (dev < 0 || dev >= 64) dev = 0;
    if (!cached[dev]) {
        int sms = 0, per_sm = 0, per_sm2 = 0;
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_hop_odd<true, EPI_SHIFT>, HOP_THREADS, 0);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm2, k_hop_even<true>, HOP_THREADS, 0);
        per_sm = per_sm < per_sm2 ? per_sm : per_sm2;
        if (sms <= 0) sms = 152;
        if (per_sm <= 0) per_sm = 1;
        cached[dev] = sms * per_sm;
    }
    int want = (g.Vh + HOP_THREADS - 1) / HOP_THREADS;
    return want < cached[dev] ? want : cached[dev];
}

void launch_hop_even_f32(const Geom &g, const SiteTerm &st, const float2 *links, const float2 *psi_o, float2 *t_e,
                         bool dag, cudaStream_t s) {
    const int nb = hop_blocks_f32(g), chunk = (g.Vh + nb - 1) / nb;
    if (dag)
        k_hop_even<true><<<nb, HOP_THREADS, 0, s>>>(g, st, links, psi_o, t_e, chunk);
    else
        k_hop_even<false><<<nb, HOP_THREADS, 0, s>>>(g, st, links, psi_o, t_e, chunk);
}

void launch_hop_odd_f32(const Geom &g, const SiteTerm &st, const float2 *links, const float2 *psi_o,
                        const float2 *t_e, float2 *y_o, bool dag, HopEpi epi, const HopEpiArgsF &ea, cudaStream_t s) {
    const int nb = hop_blocks_f32(g), chunk = (g.Vh + nb - 1) / nb;
#define TMND_ODD32(D, E) k_hop_odd<D, E><<<nb, HOP_THREADS, 0, s>>>(g, st, links, psi_o, t_e, y_o, ea, chunk)
    if (epi == EPI_STORE) {
        dag ? TMND_ODD32(true, EPI_STORE) : TMND_ODD32(false, EPI_STORE);
    } else {
        TMND_ODD32(true, EPI_SHIFT);  // of Qhat^2 + sigma only
    }
#undef TMND_ODD32
}
