// Sums of a few doubles on the integer pipes.  GB300 issues 2 FP64 operations a
// clock and SM and 64 to 128 integer ones, so a neighbour sum is cheaper with the
// significands aligned to the largest exponent and added as 64-bit integers:
// kFxGuard bits are kept below the last place of the largest term, an addend
// loses less than 2^-kFxGuard of that place (an FP64 addition up to half of it),
// and the sum is rounded once.  Up to 2^(10 - kFxGuard) = 16 terms fit.
#pragma once
#include <cstdint>

namespace plhr {

constexpr int kFxGuard = 6;

struct FxTerm {
    unsigned a;   // upper word of |x|: exponent (11 bits), 20 bits of the significand
    unsigned s;   // 0 or ~0: the sign
    uint64_t m;   // significand with its leading one, shifted up by kFxGuard
};

__device__ __forceinline__ FxTerm fx_term(double x) {
    const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
    FxTerm t;
    t.a = hi & 0x7fffffffu;
    t.s = (unsigned)((int)hi >> 31);
    const unsigned mh = (hi & 0xfffffu) | 0x100000u;
    t.m = (uint64_t)__funnelshift_l(lo, mh, kFxGuard) << 32 | (lo << kFxGuard);
    return t;
}

// t aligned to the exponent of top (upper words with the low 20 bits set): the
// value's one's complement where it is negative, its sign to be subtracted.
// Terms 2^64 below the largest, zeros and subnormals among them, are 0 (shr
// clamps its amount).
__device__ __forceinline__ uint64_t fx_align(const FxTerm& t, unsigned top) {
    uint64_t v;
    asm("shr.u64 %0, %1, %2;" : "=l"(v) : "l"(t.m), "r"((top - t.a) >> 20));
    return v ^ ((uint64_t)t.s << 32 | t.s);
}

// Exponents for which the aligned sum and its scale are normal numbers: largest
// terms from 2^-400 to 2^400.  Everything else (zeros only, infinities, NaN)
// takes FP64 operations.
__device__ __forceinline__ bool fx_in_range(unsigned top) { return (top >> 20) - 623u <= 800u; }

// c 2^(exponent of the sums aligned to top); |c| between 2^-500 and 2^500
__device__ __forceinline__ double fx_scale(double c, unsigned top) {
    return __hiloint2double(__double2hiint(c) + (((int)(top >> 20) - 1075 - kFxGuard) << 20), __double2loint(c));
}
inline bool fx_scale_ok(double c) {
    const double a = c < 0.0 ? -c : c;
    return a >= 0x1p-500 && a <= 0x1p500;
}

// 64-bit integer to double, rounded once: (2^84 + 2^63 + 2^32 hi) and (2^52 + lo)
// put together from their words, the first difference exact
__device__ __forceinline__ double fx_double(int64_t v) {
    const int hi = (int)((uint64_t)v >> 32), lo = (int)(uint32_t)(uint64_t)v;
    const double h = __hiloint2double(0x45300000, (int)((unsigned)hi ^ 0x80000000u));
    const double l = __hiloint2double(0x43300000, lo);
    return (h - (0x1p84 + 0x1p63 + 0x1p52)) + l;
}

// A grid with x fastest, in rows of a block; neighbours outside are 0 or wrap around
struct FxBox {
    int64_t nx, ny, nz;
    int periodic;
};

// Points that a thread of fx_walk takes, 0 where the FP64 kernels stay: small
// blocks are bound by latency, and longer walks leave too few threads (128^3 x 16:
// 515 us in FP64, 435 / 339 / 287 / 261 / 249 / 244 at 1 / 2 / 4 / 8 / 16 / 32 points;
// 64^3 x 5: 27 in FP64, 23 / 21 / 23 / 25 at 2 / 4 / 8 / 16; 24^3 x 16: 11, 9 / 11 at 2 / 4).
inline int fx_planes(int d, const FxBox& g, int nc, double coef) {
    const int64_t elems = g.nx * g.ny * g.nz * nc, n = d == 3 ? g.nz : g.ny;
    if (elems < 500000 || !fx_scale_ok(coef)) return 0;
    int64_t p = elems / 400000;
    p = p < 2 ? 2 : p > 16 ? 16 : p;
    if (p > n) p = n;
    if (g.nx * nc > (int64_t)1 << 30 || (d == 3 && g.ny > 65535) || (n + p - 1) / p > 65535) return 0;
    return (int)p;
}
constexpr int kFxThreads = 256;
inline dim3 fx_grid(int d, const FxBox& g, int nc, int planes) {
    const int64_t n = d == 3 ? g.nz : g.ny;
    return dim3((unsigned)((g.nx * nc + kFxThreads - 1) / kFxThreads), (unsigned)(d == 3 ? g.ny : 1),
                (unsigned)((n + planes - 1) / planes));
}

// Calls f(row, column, x_c, coef * s) for the points of this thread, `planes` up the
// slowest axis (z, or y in 2D): s is the sum of x_c's neighbours or, with LAP,
// 2d x_c minus it.  A thread keeps the terms below, at and above it; the other
// neighbours come from the caches.
template <bool D3, bool LAP, class F>
__device__ __forceinline__ void fx_walk(const FxBox& g, int nc, int planes, double coef, const double* __restrict__ x,
                                        int64_t ldx, F&& f) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int)g.nx * nc) return;
    const int ix = t / nc, c = t - ix * nc, iy = D3 ? blockIdx.y : 0;
    const int n = (int)(D3 ? g.nz : g.ny);
    const int w0 = blockIdx.z * planes, w1 = w0 + planes < n ? w0 + planes : n;
    const int64_t sz = g.nx * g.ny, step = D3 ? sz : g.nx, dw = ldx * step;
    const bool per = g.periodic;
    const bool bx0 = ix > 0 || per, bx1 = ix < g.nx - 1 || per;
    const bool by0 = D3 && (iy > 0 || per), by1 = D3 && (iy < g.ny - 1 || per);
    const int64_t dx0 = ldx * (ix > 0 ? -1 : g.nx - 1), dx1 = ldx * (ix < g.nx - 1 ? 1 : -(g.nx - 1));
    const int64_t dy0 = ldx * (iy > 0 ? -g.nx : sz - g.nx), dy1 = ldx * (iy < g.ny - 1 ? g.nx : g.nx - sz);
    int64_t row = (int64_t)w0 * step + (int64_t)iy * g.nx + ix;
    const double* xp = x + row * ldx + c;
    double xc = xp[0], xb = w0 > 0 ? xp[-dw] : per ? xp[(int64_t)(n - 1) * dw] : 0.0;
    FxTerm tb = fx_term(xb), tc = fx_term(xc);
    for (int p = w0; p < w1; ++p) {
        const double xu = p + 1 < n ? xp[dw] : per ? xp[-(int64_t)(n - 1) * dw] : 0.0;
        const double x0 = bx0 ? xp[dx0] : 0.0, x1 = bx1 ? xp[dx1] : 0.0;
        const double y0 = by0 ? xp[dy0] : 0.0, y1 = by1 ? xp[dy1] : 0.0;
        const FxTerm tu = fx_term(xu), u0 = fx_term(x0), u1 = fx_term(x1), v0 = fx_term(y0), v1 = fx_term(y1);
        unsigned top = max(max(max(tb.a, tu.a), u0.a), u1.a);
        if (D3) top = max(max(top, v0.a), v1.a);
        if (LAP) top = max(top, tc.a);
        top |= 0xfffffu;
        double v;
        if (fx_in_range(top)) {
            uint64_t s = fx_align(tb, top) + fx_align(tu, top) + fx_align(u0, top) + fx_align(u1, top);
            unsigned neg = tb.s + tu.s + u0.s + u1.s;
            if (D3) {
                s += fx_align(v0, top) + fx_align(v1, top);
                neg += v0.s + v1.s;
            }
            s -= (uint64_t)(int64_t)(int)neg;
            if (LAP) s = (D3 ? 6u : 4u) * (fx_align(tc, top) + (tc.s & 1u)) - s;
            v = fx_scale(coef, top) * fx_double((int64_t)s);
        } else {
            v = D3 ? ((x0 + x1) + (y0 + y1)) + (xb + xu) : (x0 + x1) + (xb + xu);
            if (LAP) v = fma(D3 ? 6.0 : 4.0, xc, -v);
            v *= coef;
        }
        f(row, c, xc, v);
        tb = tc;
        tc = tu;
        xb = xc;
        xc = xu;
        xp += dw;
        row += step;
    }
}

}  // namespace plhr
