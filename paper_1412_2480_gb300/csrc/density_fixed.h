// A particle's contributions to the charge density as whole numbers: device code that also
// compiles for the host, where a test compares it with exact arithmetic.
//
// Offsets are FP32 numbers in [0, 1); those that are whole multiples F of 2^-31 (all from 2^-8
// on, and zero) have weights that are short polynomials of F, exact in a few 32-bit products.
// A contribution, the product of one weight per axis, comes as three words: a whole number of
// 2^-62 at order 1 (exact) and of 2^-88 at orders 2 and 3, there of 3/2 weights each (all of
// them multiples of fourths then). It is off by 2^-53.5 of itself at most, however small it is:
// a particle with a contribution below about 2^-34 is refused, as are other offsets.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define PIC_DENS __device__ __forceinline__
#else
#define PIC_DENS inline
#endif

namespace pic {

typedef unsigned long long u64;

PIC_DENS int clz32(unsigned x) {  // 32 of 0
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}
PIC_DENS unsigned funnel_right(unsigned lo, unsigned hi, int s) {  // 0 <= s <= 31
#ifdef __CUDA_ARCH__
    return __funnelshift_r(lo, hi, s);
#else
    return (unsigned)((((u64)hi << 32) | lo) >> s);
#endif
}

// The offset with these bits as F 2^-31.
PIC_DENS bool fixed_offset(unsigned bits, unsigned& F) {
    const int sh = (int)(bits >> 23) - 119;
    F = sh < 0 ? 0u : ((bits & 0x7fffffu) | 0x800000u) << sh;
    return sh >= 0 || bits == 0u;
}

// A number of three words, least significant first.
struct Words {
    unsigned w[3];
};
PIC_DENS Words words_sub(const Words& a, const Words& b) {
    Words r;
#ifdef __CUDA_ARCH__
    asm("sub.cc.u32 %0, %3, %6;\n subc.cc.u32 %1, %4, %7;\n subc.u32 %2, %5, %8;\n"
        : "=r"(r.w[0]), "=r"(r.w[1]), "=r"(r.w[2])
        : "r"(a.w[0]), "r"(a.w[1]), "r"(a.w[2]), "r"(b.w[0]), "r"(b.w[1]), "r"(b.w[2]));
#else
    const unsigned __int128 x = ((unsigned __int128)a.w[2] << 64) | ((u64)a.w[1] << 32) | a.w[0];
    const unsigned __int128 y = ((unsigned __int128)b.w[2] << 64) | ((u64)b.w[1] << 32) | b.w[0];
    const unsigned __int128 d = x - y;
    r.w[0] = (unsigned)d;
    r.w[1] = (unsigned)(d >> 32);
    r.w[2] = (unsigned)(d >> 64);
#endif
    return r;
}

// ---- order 2 ----------------------------------------------------------------------------
// The outer weights are h^2 / 2 and g^2 / 2, h the distance of the offset from the upper edge
// of the nearest node's cell, g = 1 - h the one from its lower edge. Corners are exact products
// of them, cut off below 2^-88. What is left of a row or column follows by subtraction from its
// outer weight, whose products with the axis across add up to it: a particle's charge is exact,
// and as cut numbers are subtracted nothing comes out below zero.

PIC_DENS void quadratic_ends(unsigned F, bool& up, unsigned& H, unsigned& G) {
    constexpr unsigned one = 1u << 31;
    up = F >= one / 2;
    H = (up ? one + one / 2 : one / 2) - F;
    G = one - H;
}
PIC_DENS unsigned least_nonzero(unsigned a, unsigned b) { return b == 0u ? a : (a < b ? a : b); }  // a > 0

// x y 2^-38, x and y squares of H or G
PIC_DENS Words corner_words(u64 x, u64 y) {
    const unsigned x0 = (unsigned)x, x1 = (unsigned)(x >> 32), y0 = (unsigned)y, y1 = (unsigned)(y >> 32);
    const u64 t = (u64)x0 * y0;
    const u64 u = (u64)x1 * y0 + (t >> 32);
    const u64 v = (u64)x0 * y1 + (unsigned)u;
    const u64 w = (u64)x1 * y1 + (u >> 32) + (v >> 32);
    const unsigned a = (unsigned)v, b = (unsigned)w, c = (unsigned)(w >> 32);
    return Words{{funnel_right(a, b, 6), funnel_right(b, c, 6), c >> 6}};
}
// a square of H or G, halved, as a number of 2^-88
PIC_DENS Words end_words(u64 x) {
    const unsigned l = (unsigned)x, h = (unsigned)(x >> 32);
    return Words{{l << 25, funnel_right(l, h, 7), h >> 7}};
}

// ---- order 3 ----------------------------------------------------------------------------
// 3/2 of the weights: f^3 / 4 (the outermost on f's side), as m 2^-63 2^-s with the leading bits
// of m set, and 1 - 3/2 f^2 + 3/4 f^3 = c 2^-63 on the other side of the middle.
PIC_DENS void cubic(unsigned F, u64& m, int& s, u64& c) {
    const int n = F ? clz32(F) : 0;
    const unsigned a = F << n;
    const u64 a2 = (u64)a * a, f2 = (u64)F * F;
    m = (u64)(unsigned)(a2 >> 32) * a + ((u64)(unsigned)a2 * a >> 32);
    s = 3 * n;
    const u64 f3 = (u64)(unsigned)(f2 >> 32) * F + ((u64)(unsigned)f2 * F >> 32);  // f^3 / 4
    c = (1ull << 63) - 3 * (f2 - f3);
}

// The product's upper 64 bits: the lower halves' product is left out and 3/4 added in its
// place, so the result is off by -5/4 to 3/4.
PIC_DENS u64 mul_hi(u64 x, u64 y) {
    const unsigned x0 = (unsigned)x, x1 = (unsigned)(x >> 32), y0 = (unsigned)y, y1 = (unsigned)(y >> 32);
    const u64 t = (u64)x1 * y0 + 0xC0000000ull;
    const u64 u = (u64)x0 * y1 + (unsigned)t;
    return (u64)x1 * y1 + (t >> 32) + (u >> 32);
}
// p 2^-62 2^-s as a number of 2^-88, s <= 31
PIC_DENS Words shifted_words(u64 p, int s) {
    const unsigned lo = (unsigned)p << 26, mid = (unsigned)(p >> 6), hi = (unsigned)(p >> 38);
    return Words{{funnel_right(lo, mid, s), funnel_right(mid, hi, s), hi >> s}};
}

// The contributions of a particle in cell (i, j) with offsets Fx, Fy: add(bx, by, r, v) for
// every row by + r of P + 1 nodes from bx. false, and nothing added: refused.
template <int P, typename Add>
PIC_DENS bool density_contributions(int i, unsigned Fx, int j, unsigned Fy, Add&& add) {
    if constexpr (P == 1) {
        const u64 xy = (u64)Fx * Fy, x = (u64)Fx << 31, y = (u64)Fy << 31;
        const auto row = [&](int r, u64 a, u64 b) {
            const Words v[2] = {{{(unsigned)a, (unsigned)(a >> 32), 0u}}, {{(unsigned)b, (unsigned)(b >> 32), 0u}}};
            add(i, j, r, v);
        };
        row(0, (1ull << 62) - x - y + xy, x - xy);
        row(1, y - xy, xy);
        return true;
    } else if constexpr (P == 2) {
        bool ux, uy;
        unsigned Hx, Gx, Hy, Gy;
        quadratic_ends(Fx, ux, Hx, Gx);
        quadratic_ends(Fy, uy, Hy, Gy);
        // the smallest corner, (l l')^2 / 4, below 2^-34
        if ((u64)least_nonzero(Hx, Gx) * least_nonzero(Hy, Gy) < 1ull << 46) return false;
        const int bx = ux ? i : i - 1, by = uy ? j : j - 1;
        const u64 x0 = (u64)Hx * Hx, x2 = (u64)Gx * Gx;
        Words m0 = end_words(x0), m2 = end_words(x2), yc{{0u, 0u, 1u << 24}};
#pragma unroll
        for (int b = 0; b <= 2; b += 2) {
            const u64 y = b ? (u64)Gy * Gy : (u64)Hy * Hy;
            const Words e = end_words(y);
            Words v[3];
            v[0] = corner_words(x0, y);
            v[2] = corner_words(x2, y);
            v[1] = words_sub(words_sub(e, v[0]), v[2]);
            m0 = words_sub(m0, v[0]);
            m2 = words_sub(m2, v[2]);
            yc = words_sub(yc, e);
            add(bx, by, b, v);
        }
        const Words v[3] = {m0, words_sub(words_sub(yc, m0), m2), m2};
        add(bx, by, 1, v);
        return true;
    } else {
        // [0]: the offset from the cell's lower node, f; [1]: 1 - f
        u64 mx[2], my[2], cx[2], cy[2];
        int sx[2], sy[2];
        cubic(Fx, mx[0], sx[0], cx[0]);
        cubic((1u << 31) - Fx, mx[1], sx[1], cx[1]);
        cubic(Fy, my[0], sy[0], cy[0]);
        cubic((1u << 31) - Fy, my[1], sy[1], cy[1]);
        if ((sx[0] > sx[1] ? sx[0] : sx[1]) + (sy[0] > sy[1] ? sy[0] : sy[1]) > 31) return false;
        const u64 X[4] = {mx[1], cx[0], cx[1], mx[0]}, Y[4] = {my[1], cy[0], cy[1], my[0]};
        const int SX[4] = {sx[1], 0, 0, sx[0]}, SY[4] = {sy[1], 0, 0, sy[0]};
#pragma unroll
        for (int b = 0; b < 4; b++) {
            Words v[4];
#pragma unroll
            for (int a = 0; a < 4; a++) v[a] = shifted_words(mul_hi(X[a], Y[b]), SX[a] + SY[b]);
            add(i - 1, j - 1, b, v);
        }
        return true;
    }
}

}  // namespace pic
