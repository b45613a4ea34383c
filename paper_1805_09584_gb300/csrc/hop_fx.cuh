// FP64-accurate vectors and links in two-digit fixed point, for the integer stencil (hop_fx.cu).
//
// GB300 has 2 FP64 multiply-adds per clock and SM, but 30 integer ones of the form
// 32 x 32 + 64 -> 64 bits (both measured).  A real number is kept as q 2^(E - 56) with an
// integer |q| <= 2^56, q = h 2^28 + l (h, l signed 32-bit words, |h| <= 2^28, -2^27 <= l < 2^27):
//   spinors: one exponent E per site, all 24 components below 2^E in magnitude, so the format
//            carries 56 bits below the largest component of the site (a double has 53);
//   links:   E = 0 (|U_ij| <= 1), the antiperiodic sign of the time boundary folded in.
// A product's 2^-56 part costs three integer multiply-adds, h h, h l and l h, the last two into
// an accumulator of their own; l l is below 2^-58 of the largest term and is left out.
#pragma once

#include "tmnd_internal.cuh"

// Spinor in HBM: blocks of 16 consecutive half-lattice sites, each 24 runs (one per component) of 16
// words (re.h, re.l, im.h, im.l); then V/2 exponents.  A component is a constant distance from its
// site's first word, so one address serves a site, and a run is two whole 128-byte lines.  Links of one
// parity and direction: the same with 9 runs per block.
struct FxIn {
    const int4 *q;
    const int *e;
};
struct FxOut {
    int4 *q;
    int *e;
};
constexpr int FX_ZERO = -(1 << 20);  // exponent of a site whose components are all zero
constexpr int FX_NAN = 1 << 20;      // exponent of a site that holds, or met, a NaN or an infinity

FxSite fx_site(const SiteTerm &st);

// Epilogue of the odd kernel on y = A psi - H t
enum FxEpi {
    FX_STORE = 0,        // out = y (digits)
    FX_STORE_NORMS = 1,  // out = y (digits); partials |y|^2, |psi|^2
    FX_F64 = 2,          // out64 = y
    FX_F64_QHAT = 3,     // out64 = gamma_5 tau_1 y
    FX_F64_SHIFT = 4,    // out64 = y + sigma aux64
    FX_RESID = 5,        // r = b64 - y - sigma aux64; partial |r|^2
    FX_MMS_R = 6         // r = r_in - alpha (y + sigma p); partial |r|^2
};
struct FxOdd {
    FxOut out;
    double2 *out64;
    const double2 *aux64, *b64;
    double sigma;
    FxIn p;                 // FX_MMS_R: the vector multiplied by sigma
    int2 sig;               // sigma's digits and exponent (set by the launcher)
    int sig_e;
    const double2 *r_in;
    double2 *r;
    const double *alpha;    // FX_MMS_R: device scalar
    double *part_out;       // partial sums, one (FX_STORE_NORMS: two) per block
    const int *done;        // if non-null and *done != 0 the kernel returns immediately
};

constexpr int FX_THREADS = 128;  // four warps, one per direction mu, on 16 sites at a time
constexpr int FX_BLOCKS = 5;     // resident blocks of that size per SM

// Several right-hand sides in one launch (the grid's y): distance of their fixed-point vectors in bytes
// and of their FP64 vectors in complex numbers.
struct FxBatch {
    int nrhs = 1;
    size_t stride = 0;
    size_t n64 = 0;
};

int fx_blocks(const Geom &g);  // blocks (= reduction partials) of every stencil launch on this lattice
void launch_fx_from_f64(const Geom &g, const double2 *in, FxOut out, cudaStream_t s, const FxBatch &bt = FxBatch());
void launch_fx_to_f32(const Geom &g, double a, FxIn in, float2 *out, cudaStream_t s);  // out = a in
void launch_fx_pack_links(const Geom &g, const double2 *canon, int4 *out, cudaStream_t s);
// p = r + beta p unless *skip
void launch_fx_pupdate(const Geom &g, const int *skip, const double *beta, const double2 *r, FxOut p, cudaStream_t s);
void launch_fx_even(const Geom &g, const FxSite &st, const int4 *links, FxIn psi, FxOut out, bool dag,
                    const int *done, cudaStream_t s, const FxBatch &bt = FxBatch());
// ea.out may be psi's own buffer (FX_STORE): a block reads its run's psi before it writes the run
void launch_fx_odd(const Geom &g, const FxSite &st, const int4 *links, FxIn psi, FxIn te, bool dag, FxEpi epi,
                   FxOdd ea, cudaStream_t s, const FxBatch &bt = FxBatch());
// Right-hand sides per launch of an operator application: more than one only while a launch has less work
// than two rounds of blocks, so that the temporaries (2 fx_bytes each) stay small.
int fx_batch(const Geom &g, int nrhs);

constexpr int FX_RUN = 16;
// first word of site h (component c at + c FX_RUN), for ncomp components per site
__host__ __device__ inline int fx_at(int h, int ncomp) { return (h >> 4) * (ncomp * FX_RUN) + (h & 15); }
__host__ __device__ inline size_t fx_sites(int Vh) { return ((size_t)Vh + 15) & ~(size_t)15; }
inline size_t fx_link_words(int Vh) { return 2 * 4 * 9 * fx_sites(Vh); }
inline size_t fx_bytes(int Vh) {
    return (fx_sites(Vh) * (NCOMP * sizeof(int4) + sizeof(int)) + 255) & ~(size_t)255;
}
inline FxOut fx_out(void *base, int Vh) {
    return FxOut{(int4 *)base, (int *)((char *)base + fx_sites(Vh) * NCOMP * sizeof(int4))};
}
// the spinor `bytes` further on
__host__ __device__ inline FxIn fx_next(FxIn v, size_t bytes) {
    return FxIn{(const int4 *)((const char *)v.q + bytes), (const int *)((const char *)v.e + bytes)};
}
__host__ __device__ inline FxOut fx_next(FxOut v, size_t bytes) {
    return FxOut{(int4 *)((char *)v.q + bytes), (int *)((char *)v.e + bytes)};
}
inline FxIn fx_in(FxOut o) { return FxIn{o.q, o.e}; }

// --------------------------------------------------------- device helpers
__device__ __forceinline__ bool fx_is_nan(int e) { return e > FX_NAN / 2; }

// 2^k as a double, k within the normal range
__device__ __forceinline__ double fx_pow2(int k) { return __hiloint2double((k + 1023) << 20, 0); }

// Factor(s) that turn an integer word into the double it stands for: 2^k, NaN for a NaN site.
// Where 2^k is no normal number (fields near the ends of the FP64 range) it is split in two.
struct FxScale {
    double s1, s2;
    bool split;
};
__device__ __forceinline__ FxScale fx_scale(int e, int k) {
    FxScale r;
    r.split = k < -1000 || k > 960;
    r.s2 = 1.0;
    if (fx_is_nan(e)) {
        r.s1 = __longlong_as_double(0x7ff8000000000000ll);
        r.split = false;
    } else if (!r.split) {
        r.s1 = fx_pow2(k);
    } else {
        const int a = max(min(k, 2000), -2000) / 2, b = max(min(k, 2000), -2000) - a;
        r.s1 = fx_pow2(a);
        r.s2 = fx_pow2(b);
    }
    return r;
}
__device__ __forceinline__ double fx_to_double(long long v, const FxScale &s) {
    double d = (double)v * s.s1;
    if (s.split) d *= s.s2;
    return d;
}
__device__ __forceinline__ long long fx_word(int h, int l) { return (long long)h * (1 << 28) + l; }

// word with |v| <= 2^56 -> its digits
__device__ __forceinline__ void fx_split(long long v, int &h, int &l) {
    const long long t = v + (1ll << 27);
    h = (int)(t >> 28);
    l = ((int)t & 0x0fffffff) - (1 << 27);
}

// A warp holds 16 consecutive sites: lanes 0..15 the first flavour, 16..31 the second.
// Twelve complex doubles of one flavour of a site -> digits, exponent common to both flavours.
__device__ __forceinline__ void fx_from_doubles(const double2 v[12], int4 q[12], int &e) {
    int mx = 0, nz = 0;
#pragma unroll
    for (int c = 0; c < 12; c++) {
        const int a = __double2hiint(v[c].x) & 0x7fffffff, b = __double2hiint(v[c].y) & 0x7fffffff;
        mx = max(mx, max(a, b));
        nz |= __double2loint(v[c].x) | __double2loint(v[c].y);
    }
    mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
    nz |= __shfl_xor_sync(0xffffffffu, nz, 16);
    const int ef = max(mx >> 20, 1);  // exponent field of the largest component (subnormals: 1)
    const bool bad = (mx >> 20) == 0x7ff;
    e = bad ? FX_NAN : (mx | nz) == 0 ? FX_ZERO : ef - 1022;
    auto conv = [&](double x, int &h, int &l) {
        const int hw = __double2hiint(x), lw = __double2loint(x);
        const int ex = (hw >> 20) & 0x7ff;
        const unsigned mh = (unsigned)(hw & 0xfffff) | (ex ? 0x100000u : 0u);
        const int r = min(ef - max(ex, 1), 63);
        const unsigned long long w = (((unsigned long long)mh << 37) | ((unsigned long long)(unsigned)lw << 5)) >> r;
        const long long sg = (long long)(hw >> 31);
        // (+-w + rounding half + 2^27 of the digit split) at two bits below the word's unit
        const long long t = ((long long)w ^ sg) + ((2ll + (1ll << 29)) - sg);
        h = bad ? 0 : (int)(t >> 30);
        l = bad ? 0 : (int)((unsigned)t >> 2 & 0x0fffffff) - (1 << 27);
    };
#pragma unroll
    for (int c = 0; c < 12; c++) {
        conv(v[c].x, q[c].x, q[c].y);
        conv(v[c].y, q[c].z, q[c].w);
    }
}
