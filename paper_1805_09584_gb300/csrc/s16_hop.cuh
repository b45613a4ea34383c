// Arithmetic of the sloppy stencil (FP32 on 16-bit storage, kernels in s16_kernels.cuh): decoding, the
// per-direction link products and accumulation.
//
// One thread per site and flavour.  The two spins of a projected half spinor share every link entry, so each
// pair lives in one float2 and link products, projections and accumulations are packed f32x2 instructions.
// Decoding is one byte permute per value (the float 2^23 + 32768 + n); the spin projection u -+ B l is formed
// from two decoded floats exactly (their difference, or (u - 2 bias) + l), so the projected half spinor is
// exact before the link is applied.  The neighbour's scale nrm/32767 enters as one factor of the
// accumulation; the antiperiodic sign sits in the decoded link.
#pragma once

#include "tmnd_internal.cuh"

namespace {

constexpr float INV_QMAX = 1.0f / S16_QMAX;

using f2 = float2;  // (spin 0, spin 1)

__device__ __forceinline__ f2 dup(float a) { return make_float2(a, a); }
// -a by flipping the sign bit on the integer pipe (keeps the FP32 pipe for products)
__device__ __forceinline__ float fneg(float a) { return __int_as_float(__float_as_int(a) ^ (int)0x80000000); }
__device__ __forceinline__ f2 add2(f2 a, f2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ f2 mul2(f2 a, f2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ S16In s16_at(S16In a, size_t off) {
    return S16In{(const int4 *)((const char *)a.q + off), (const float *)((const char *)a.nrm + off)};
}
__device__ __forceinline__ S16Out s16_at(S16Out a, size_t off) {
    return S16Out{(int4 *)((char *)a.q + off), (float *)((char *)a.nrm + off)};
}

// one flavour of a neighbour: its 12 words and its scale
struct Raw {
    int4 q[3];
    float nrm;
};
__device__ __forceinline__ int word(const Raw &r, int k) {
    const int4 &v = r.q[k / 4];
    return k % 4 == 0 ? v.x : k % 4 == 1 ? v.y : k % 4 == 2 ? v.z : v.w;
}
__device__ __forceinline__ void load_raw(const S16In &in, int f, int h, Raw &r) {
    const int4 *q = in.q + s16_qi(f * 3, h);
#pragma unroll
    for (int j = 0; j < 3; j++) r.q[j] = q[j * S16_BLOCK_SITES];
    r.nrm = in.nrm[s16_ni(h)];
}
__device__ __forceinline__ void load_raw2(const S16In &in, int h, Raw r[2]) {  // both flavours
    const int4 *q = in.q + s16_qi(0, h);
#pragma unroll
    for (int j = 0; j < 6; j++) r[j / 3].q[j % 3] = q[j * S16_BLOCK_SITES];
    r[0].nrm = r[1].nrm = in.nrm[s16_ni(h)];
}

// (u.x + SX l.x, u.y + SY l.y) for biased floats u, l (exact integer results)
template <int SX, int SY>
__device__ __forceinline__ f2 comb(f2 u, f2 l) {
    if (SX < 0 && SY < 0) return fma2(l, dup(-1.0f), u);
    const f2 v = add2(u, make_float2(SX > 0 ? -2.0f * S16_DEC_BIAS : 0.0f, SY > 0 ? -2.0f * S16_DEC_BIAS : 0.0f));
    return SX > 0 && SY > 0 ? add2(v, l) : fma2(l, make_float2((float)SX, (float)SY), v);
}

// A link's words: rows 0 and 1, scale 32767
__device__ __forceinline__ void load_link(const int2 *__restrict__ L, int h, int wv[6]) {
#pragma unroll
    for (int j = 0; j < 3; j++) {
        int2 w;
        asm("ld.global.nc.L1::no_allocate.v2.s32 {%0, %1}, [%2];" : "=r"(w.x), "=r"(w.y) : "l"(&L[s16_li(j, h)]));
        wv[2 * j] = w.x;
        wv[2 * j + 1] = w.y;
    }
}
// Decode a link and rebuild row 2 = conj(row 0 x row 1) (det U = 1) as integer-valued floats at that scale,
// times sg (+-1).  u: 9 complex numbers, row-major.
__device__ __forceinline__ void decode_link(const int wv[6], float sg, f2 u[9]) {
#pragma unroll
    for (int k = 0; k < 6; k++) u[k] = make_float2(s16_lo(wv[k]), s16_hi(wv[k]));
#pragma unroll
    for (int k = 0; k < 3; k++) {
        const f2 a1 = u[(k + 1) % 3], a2 = u[(k + 2) % 3], b1 = u[3 + (k + 1) % 3], b2 = u[3 + (k + 2) % 3];
        float re = fmaf(a1.x, b2.x, -a1.y * b2.y);
        float im = fmaf(a1.x, b2.y, a1.y * b2.x);
        re = fmaf(-a2.x, b1.x, fmaf(a2.y, b1.y, re));
        im = fmaf(-a2.x, b1.y, fmaf(-a2.y, b1.x, im));
        u[6 + k] = make_float2(re * INV_QMAX, -im * INV_QMAX);
    }
#pragma unroll
    for (int k = 0; k < 9; k++) u[k] = make_float2(sg * u[k].x, sg * u[k].y);
}

// Decoded links of a block's sites in shared memory: per direction four float4 planes (8 complex) and a
// float2 plane (the ninth).
template <int SITES>
struct LinkTile {
    float4 a[8][4][SITES];
    float2 b[8][SITES];
    __device__ __forceinline__ void put(int d, int i, const f2 u[9]) {
#pragma unroll
        for (int q = 0; q < 4; q++) a[d][q][i] = make_float4(u[2 * q].x, u[2 * q].y, u[2 * q + 1].x, u[2 * q + 1].y);
        b[d][i] = u[8];
    }
    __device__ __forceinline__ void get(int d, int i, f2 u[9]) const {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const float4 v = a[d][q][i];
            u[2 * q] = make_float2(v.x, v.y);
            u[2 * q + 1] = make_float2(v.z, v.w);
        }
        u[8] = b[d][i];
    }
};

// Hop of direction MU, DIR into acc: up[colour][re, im] the pair of spins 0, 1; lo the pair 2, 3.
template <int MU, int DIR, bool G5IN, bool FIRST>
__device__ __forceinline__ void hop_dir(const Raw &r, const f2 u[9], f2 up[3][2], f2 lo[3][2]) {
    // projection chi = u -+ B l (upper spins 0, 1), exact integers.
    // B l, by direction (lower spin index, components):
    //   MU 0: lower 2+s,   (-l.re, -l.im)
    //   MU 1: lower 3-s,   (l.im, -l.re)
    //   MU 2: lower 3-s,   s = 0: (-l.re, -l.im); s = 1: (l.re, l.im)
    //   MU 3: lower 2+s,   s = 0: (l.im, -l.re);  s = 1: (-l.im, l.re)
    constexpr bool plus = (DIR < 0) != G5IN;
    constexpr int P = plus ? 1 : -1;
    constexpr bool swap = MU == 1 || MU == 2;
    f2 chr[3], chi[3];
#pragma unroll
    for (int c = 0; c < 3; c++) {
        const int u0 = word(r, c), u1 = word(r, 3 + c);
        const int l0 = word(r, swap ? 9 + c : 6 + c), l1 = word(r, swap ? 6 + c : 9 + c);
        const f2 uR = make_float2(s16_flo(u0), s16_flo(u1)), uI = make_float2(s16_fhi(u0), s16_fhi(u1));
        const f2 lR = make_float2(s16_flo(l0), s16_flo(l1)), lI = make_float2(s16_fhi(l0), s16_fhi(l1));
        if (MU == 0) {
            chr[c] = comb<-P, -P>(uR, lR);
            chi[c] = comb<-P, -P>(uI, lI);
        } else if (MU == 1) {
            chr[c] = comb<P, P>(uR, lI);
            chi[c] = comb<-P, -P>(uI, lR);
        } else if (MU == 2) {
            chr[c] = comb<-P, P>(uR, lR);
            chi[c] = comb<-P, P>(uI, lI);
        } else {
            chr[c] = comb<P, -P>(uR, lI);
            chi[c] = comb<-P, P>(uI, lR);
        }
    }
    // v = W chi with W = U (forward) or U^+ (backward); both spins at once.
    //   forward : re = sum ur chr - sum ui chi,  im = sum ur chi + sum ui chr
    //   backward: re = sum ur' chr + sum ui' chi, im = sum ur' chi - sum ui' chr  (ur' = ur[j][i])
    const float cs = r.nrm * INV_QMAX;
    const f2 cs2 = dup(cs);
    const float cl = DIR > 0 ? -cs : cs;  // factor of the lower spins
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
        f2 a = mul2(wr[0], chr[0]);
        a = fma2(wr[1], chr[1], a);
        a = fma2(wr[2], chr[2], a);
        a = fma2(wa[0], chi[0], a);
        a = fma2(wa[1], chi[1], a);
        const f2 vr = fma2(wa[2], chi[2], a);
        f2 b = mul2(wr[0], chi[0]);
        b = fma2(wr[1], chi[1], b);
        b = fma2(wr[2], chi[2], b);
        b = fma2(wb[0], chr[0], b);
        b = fma2(wb[1], chr[1], b);
        const f2 vi = fma2(wb[2], chr[2], b);
        // upper spins += cs v; lower spins (2, 3) += cl B^+ v:
        //   MU 0: -v[s]; MU 1: (-v[1-s].im, v[1-s].re); MU 2: s = 0: v[1], s = 1: -v[0];
        //   MU 3: s = 0: (-v[0].im, v[0].re), s = 1: (v[1].im, -v[1].re)
        if (FIRST) {
            up[i][0] = mul2(cs2, vr);
            up[i][1] = mul2(cs2, vi);
            lo[i][0] = lo[i][1] = dup(0.0f);
        } else {
            up[i][0] = fma2(cs2, vr, up[i][0]);
            up[i][1] = fma2(cs2, vi, up[i][1]);
        }
        if (MU == 0) {
            lo[i][0] = fma2(dup(-cl), vr, lo[i][0]);
            lo[i][1] = fma2(dup(-cl), vi, lo[i][1]);
        } else if (MU == 1) {
            lo[i][0] = make_float2(fmaf(-cl, vi.y, lo[i][0].x), fmaf(-cl, vi.x, lo[i][0].y));
            lo[i][1] = make_float2(fmaf(cl, vr.y, lo[i][1].x), fmaf(cl, vr.x, lo[i][1].y));
        } else if (MU == 2) {
            lo[i][0] = make_float2(fmaf(cl, vr.y, lo[i][0].x), fmaf(-cl, vr.x, lo[i][0].y));
            lo[i][1] = make_float2(fmaf(cl, vi.y, lo[i][1].x), fmaf(-cl, vi.x, lo[i][1].y));
        } else {
            lo[i][0] = make_float2(fmaf(-cl, vi.x, lo[i][0].x), fmaf(cl, vi.y, lo[i][0].y));
            lo[i][1] = make_float2(fmaf(cl, vr.x, lo[i][1].x), fmaf(-cl, vr.y, lo[i][1].y));
        }
    }
}

// Quantise a site (this lane's flavour, v[spin*3 + colour]; the other flavour in lane ^ 16) and store this
// flavour's words; the first flavour's lane stores the scale.
__device__ __forceinline__ void store_site(S16Out out, int f, int h, bool on, const f2 v[12]) {
    float m = 0.0f;
#pragma unroll
    for (int k = 0; k < 12; k++) m = fmaxf(m, fmaxf(fabsf(v[k].x), fabsf(v[k].y)));
    m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, 16));
    const float sc = m > 0.0f ? S16_QMAX / m : 0.0f;
    int w[12];
#pragma unroll
    for (int k = 0; k < 12; k++) {
        const f2 e = fma2(v[k], dup(sc), dup(S16_ENC_MAGIC));
        w[k] = __byte_perm(__float_as_int(e.x), __float_as_int(e.y), 0x5410);
    }
    if (!on) return;
    if (f == 0) out.nrm[s16_ni(h)] = m * INV_QMAX;
    int4 *q = out.q + s16_qi(f * 3, h);
#pragma unroll
    for (int j = 0; j < 3; j++) q[j * S16_BLOCK_SITES] = make_int4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
}

// component k of a loaded site
__device__ __forceinline__ f2 value(const Raw &r, int k, float sc) {
    const int w = word(r, k);
    return make_float2(s16_lo(w) * sc, s16_hi(w) * sc);
}

}  // namespace
