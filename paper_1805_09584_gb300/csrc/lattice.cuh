// Neighbours of a site in the even-odd layout, with divisions by multiplication.
#pragma once

#include "tmnd_internal.cuh"

// n / d for n < 2^31 by a multiplication (Granlund and Montgomery, PLDI'94)
struct FastDiv {
    unsigned m;
    int s, d;
};
inline FastDiv fast_div(int d) {
    int s = 0;
    while ((1ll << s) < d) s++;
    return FastDiv{(unsigned)(((1ull << 32) * ((1ull << s) - (unsigned long long)d)) / (unsigned)d + 1), s, d};
}
__device__ __forceinline__ int fdiv(int n, const FastDiv &f) {
    return (int)((__umulhi((unsigned)n, f.m) + (unsigned)n) >> f.s);
}

struct LatGeom {
    int T, X, Y, Zh, Vh;
    int sx, st;               // half-index strides of x and t (y: Zh)
    FastDiv dZh, dY, dX, dsx, dst;
};
inline LatGeom lat_geom(const Geom &g) {
    const int sx = g.Zh * g.Y, st = sx * g.X;
    return LatGeom{g.T, g.X, g.Y, g.Zh, g.Vh, sx, st,
                  fast_div(g.Zh), fast_div(g.Y), fast_div(g.X), fast_div(sx), fast_div(st)};
}

// Half-indices of the two neighbours in direction MU of site h of parity P.
template <int MU, int P>
__device__ __forceinline__ void neighbours(const LatGeom &g, int h, int &hf, int &hb) {
    if (MU == 0) {
        const int t = fdiv(h, g.dst);
        hf = t + 1 == g.T ? h - (g.T - 1) * g.st : h + g.st;
        hb = t == 0 ? h + (g.T - 1) * g.st : h - g.st;
    } else if (MU == 1) {
        const int q = fdiv(h, g.dsx), x = q - fdiv(q, g.dX) * g.X;
        hf = x + 1 == g.X ? h - (g.X - 1) * g.sx : h + g.sx;
        hb = x == 0 ? h + (g.X - 1) * g.sx : h - g.sx;
    } else {
        const int r = fdiv(h, g.dZh), q = fdiv(r, g.dY), y = r - q * g.Y;
        if (MU == 2) {
            hf = y + 1 == g.Y ? h - (g.Y - 1) * g.Zh : h + g.Zh;
            hb = y == 0 ? h + (g.Y - 1) * g.Zh : h - g.Zh;
        } else {
            const int zh = h - r * g.Zh, t = fdiv(q, g.dX), x = q - t * g.X;
            const bool odd = (P + t + x + y) & 1;  // z = 2 zh + odd
            hf = !odd ? h : zh + 1 == g.Zh ? h - (g.Zh - 1) : h + 1;
            hb = odd ? h : zh == 0 ? h + (g.Zh - 1) : h - 1;
        }
    }
}

