// mm_gate_table64.h -- the FP64 path's gate table, host + device.
//
// The exponential-Euler step of a gate, x <- X + (x - X) D = x + (X - x) E,
// needs its steady state X(V) = a / (a + b) and its decay D(V) = exp(-dt (a + b))
// or E = 1 - D; for a network's fixed dt both are functions of V alone.  Evaluating the rates
// takes nine exponentials and six divisions of FP64 arithmetic per
// compartment, on a chip with two FP64 lanes per SM and clock.  The table
// holds each function as a degree-6 polynomial per 0.25 mV interval of
// +-120 mV: with u = (V - centre) / 0.25 mV in [-1/2, 1/2],
//   p(u) = c0 + u (c1 + u (c2 + u (c3 + u t(u)))),  t(u) = c4 + u (c5 + u c6),
// c0..c3 in FP64 and the tail t in FP32 (the functions vary over about 10 mV,
// so the term u^4 t is below 2^-27 of p and FP32 keeps it to 2^-50 of p).
// That is four FP64 operations per function, and one more for X: c0's rounding
// would shift X the same way everywhere in an interval, for as long as V stays
// there (it made the voltages' error after 160 steps 1.2 times the direct
// evaluation's), so the rest of c0 is kept in FP32 and added.  An interval holds E where E is at
// most 1/2 (X's rounding then enters times E) and -D elsewhere (tiny gates keep
// their relative accuracy).  The interpolation error is below FP64 rounding and
// the step's error below that of the rates evaluated directly in FP64, at the
// worst voltage and in the mean square (tests/test_gate_table64.py).
// Beyond +-120 mV the kernel evaluates the rates directly.
//
// Stored as 18 arrays of kTab64Intervals 16-byte quads (three per function:
// c0 c1 | c2 c3 | c4 c5 c6 and the rest of c0 as floats), so that the lanes of a warp, whose V lie
// close together, read adjacent quads of one array.
#pragma once
#include <stdint.h>

#include <cmath>
#include <cstring>
#include <limits>

#ifdef __CUDACC__
#define MMG_HD __host__ __device__ __forceinline__
#else
#define MMG_HD inline
#endif

namespace mmg {

constexpr int kTab64Intervals = 961;            // centres -120, -119.75, ..., 120 mV
constexpr int kTab64Funcs = 6;                  // X_m, F_m, X_h, F_h, X_n, F_n (F: E or -D)
constexpr int kTab64Quads = 3 * kTab64Funcs;
constexpr uint32_t kTab64MaxHi = 0x405E0000u;   // high word of 120.0

struct alignas(16) Quad64 {
    double a, b;
};
struct alignas(16) Quad32 {
    float a, b, c, d;
};

MMG_HD uint64_t bits(double x)
{
#ifdef __CUDA_ARCH__
    return (uint64_t)__double_as_longlong(x);
#else
    uint64_t b;
    std::memcpy(&b, &x, 8);
    return b;
#endif
}

// float <-> double by integer operations (a conversion instruction would run
// on the FP64 pipe).  narrow truncates and takes |x| <= 1/2; widen is exact
// for 0 (as 2^-127) and normal floats.
MMG_HD float narrow(double x)
{
    const uint64_t b = bits(x);
    const uint32_t hi = (uint32_t)(b >> 32), lo = (uint32_t)b, m = hi & 0x7FFFFFFFu;
    const uint32_t r = (hi & 0x80000000u) | (m >= 0x38100000u ? ((m - 0x38000000u) << 3) | (lo >> 29) : 0u);
#ifdef __CUDA_ARCH__
    return __uint_as_float(r);
#else
    float f;
    std::memcpy(&f, &r, 4);
    return f;
#endif
}

MMG_HD double widen(float x)
{
#ifdef __CUDA_ARCH__
    const uint32_t b = __float_as_uint(x);
    return __hiloint2double((int)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)), (int)(b << 29));
#else
    uint32_t b;
    std::memcpy(&b, &x, 4);
    const uint64_t d = ((uint64_t)((b & 0x80000000u) | (((b & 0x7FFFFFFFu) >> 3) + 0x38000000u)) << 32) |
                       (uint32_t)(b << 29);
    double r;
    std::memcpy(&r, &d, 8);
    return r;
#endif
}

// Whether V lies in the table (false for NaN).
MMG_HD bool in_table(double v) { return ((uint32_t)(bits(v) >> 32) & 0x7FFFFFFFu) <= kTab64MaxHi; }

struct Index64 {
    int i;     // interval
    double u;  // position in it
    float uf;  // the same, FP32
};

// Interval of V and position in it (both exact; 4 V + 480 is rounded to an
// integer by adding 3 2^51).
MMG_HD Index64 index64(double v)
{
    const double magic = 6755399441055744.0 + 480.0;
    const double t = std::fma(v, 4.0, magic);
    Index64 r;
    r.i = (int)(uint32_t)bits(t);
    r.u = std::fma(v, 4.0, -(t - magic));
    r.uf = narrow(r.u);
    return r;
}

MMG_HD double eval64(Quad64 p, Quad64 q, Quad32 s, const Index64 &t)
{
    const float tail = fmaf(fmaf(s.c, t.uf, s.b), t.uf, s.a);
    return std::fma(std::fma(std::fma(std::fma(widen(tail), t.u, q.b), t.u, q.a), t.u, p.b), t.u, p.a);
}

// The same with the rest of c0 (for X): one rounding of the exact value.
MMG_HD double eval64_rest(Quad64 p, Quad64 q, Quad32 s, const Index64 &t)
{
    const float tail = fmaf(fmaf(s.c, t.uf, s.b), t.uf, s.a);
    const double r = std::fma(std::fma(std::fma(widen(tail), t.u, q.b), t.u, q.a), t.u, p.b);
    return p.a + std::fma(r, t.u, widen(s.d));
}

// One step of a gate from its X and F (E >= 0 or -D < 0).
MMG_HD double step64(double x, double X, double F) { return std::fma(X - x, F, (int64_t)bits(F) < 0 ? X : x); }

// ---------------------------------------------------------------- builder

// Fills tab[kTab64Quads * kTab64Intervals] (16-byte entries; array k, interval
// i at k * kTab64Intervals + i) for the step dt: interpolation at the seven
// Chebyshev points of each interval, in long double.  The rates' exponentials
// at a point are products of one per interval centre and one per point.
inline void build_table64(double dt, void *tab)
{
    typedef long double LD;
    constexpr int K = 7;
    const LD pi = acosl(-1.0L), h = 0.25L;
    static const LD scale[4] = {10.0L, 18.0L, 20.0L, 80.0L};
    LD u[K], eo[K][4], ec[4], M[K][K];  // M: values at the points -> monomial coefficients in u
    for (int k = 0; k < K; ++k) {
        u[k] = k == K / 2 ? 0.0L : 0.5L * cosl(pi * (k + 0.5L) / K);
        for (int r = 0; r < 4; ++r) eo[k][r] = expl(-h * u[k] / scale[r]);
    }
    for (int k = 0; k < K; ++k) {  // Lagrange basis polynomial of point k
        LD c[K] = {1.0L}, den = 1.0L;
        int deg = 0;
        for (int j = 0; j < K; ++j) {
            if (j == k) continue;
            den *= u[k] - u[j];
            for (int d = ++deg; d > 0; --d) c[d] = c[d - 1] - u[j] * c[d];
            c[0] *= -u[j];
        }
        for (int d = 0; d < K; ++d) M[d][k] = c[d] / den;
    }
    const LD e35 = expl(-3.5L), e55 = expl(-5.5L), e40 = expl(-4.0L), e65_18 = expl(-65.0L / 18.0L),
             e65_20 = expl(-3.25L), e65_80 = expl(-65.0L / 80.0L);
    char *base = (char *)tab;
    for (int i = 0; i < kTab64Intervals; ++i) {
        const LD Vc = -120.0L + i * h;
        LD f[kTab64Funcs][K], y[3][K];
        for (int r = 0; r < 4; ++r) ec[r] = expl(-Vc / scale[r]);
        for (int k = 0; k < K; ++k) {
            const LD V = Vc + h * u[k];
            LD e[4];
            for (int r = 0; r < 4; ++r) e[r] = ec[r] * eo[k][r];
            const LD xm = -(V + 40.0L) / 10.0L, xn = -(V + 55.0L) / 10.0L;
            // x / (e^x - 1), 1 - x / 2 at x = 0
            const LD am = fabsl(xm) < 1e-9L ? 1.0L - 0.5L * xm : xm / (e[0] * e40 - 1.0L);
            const LD an = 0.1L * (fabsl(xn) < 1e-9L ? 1.0L - 0.5L * xn : xn / (e[0] * e55 - 1.0L));
            const LD bm = 4.0L * e[1] * e65_18, ah = 0.07L * e[2] * e65_20, bh = 1.0L / (1.0L + e[0] * e35),
                     bn = 0.125L * e[3] * e65_80;
            const LD a[3] = {am, ah, an}, b[3] = {bm, bh, bn};
            for (int g = 0; g < 3; ++g) {
                const LD s = a[g] + b[g];
                f[2 * g][k] = a[g] / s;
                y[g][k] = -(LD)dt * s;
            }
        }
        // F's rounding enters only times X - x: FP64's exponential is enough
        for (int g = 0; g < 3; ++g) {
            const bool e_form = y[g][K / 2] >= -0.6931471805599453L;  // E <= 1/2
            for (int k = 0; k < K; ++k) {
                const double yh = (double)y[g][k], dy = (double)(y[g][k] - yh);
                f[2 * g + 1][k] = e_form ? -(std::expm1(yh) + (LD)(std::exp(yh) * dy)) : -fabsl(std::exp(yh) * (1.0L + dy));
            }
        }
        for (int fn = 0; fn < kTab64Funcs; ++fn) {
            LD c[K];
            // differences to the centre's value: the sums are then small
            for (int d = 0; d < K; ++d) {
                c[d] = 0.0L;
                for (int k = 0; k < K; ++k)
                    if (k != K / 2) c[d] += M[d][k] * (f[fn][k] - f[fn][K / 2]);
            }
            Quad64 p{(double)f[fn][K / 2], (double)c[1]}, q{(double)c[2], (double)c[3]};
            Quad32 s{(float)c[4], (float)c[5], (float)c[6], (float)(f[fn][K / 2] - p.a)};
            // F below 2^-100 (a step far below the time constant, or far above
            // it): the tail leaves FP32's range, and widen's 2^-127 for a zero
            // could turn F's sign, which step64 goes by.  F is then its value at
            // the centre (within 2^-98 of it), all other terms zero with F's sign,
            // so that widen's 2^-127 u^4 has it too
            if (fn % 2 == 1 && std::fabs(p.a) < 0x1p-100) {
                const float z = std::copysign(0.0f, (float)p.a);
                p = Quad64{p.a == 0.0 ? std::copysign(std::numeric_limits<double>::min(), p.a) : p.a, (double)z};
                q = Quad64{(double)z, (double)z};
                s = Quad32{z, z, z, z};
            }
            const void *src[3] = {&p, &q, &s};
            for (int x = 0; x < 3; ++x)
                std::memcpy(base + 16 * ((size_t)(3 * fn + x) * kTab64Intervals + i), src[x], 16);
        }
    }
}

}  // namespace mmg
