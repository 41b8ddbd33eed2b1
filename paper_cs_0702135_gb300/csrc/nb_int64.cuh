// nb_int64.cuh -- a softened FP64 pair interaction on the integer pipes, up to
// its last multiply-adds.  The GB300's FP64 pipe completes a warp instruction
// per SM in 19.5 clocks, in which the SM can issue 78 others, and the 33 FP64
// operations of a pair kept all else idle.  Here the six differences, r^2,
// x.u, 1/r and its powers times the mass are evaluated on 62-bit significands
// (cut off, not rounded) and rounded to FP64 once: against exact arithmetic
// m/r is within 1.25, m/r^3 and b within 1.5 times 2^-53, where a chain of FP64
// operations reaches 3.3, 9 and 7.  10 FP64 operations and about 525 others
// remain (the ALU is 70 % busy, the FP64 pipe 90 %).  Plain integer code, host
// and device.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define NB_HD __host__ __device__ __forceinline__
#else
#define NB_HD inline
#include <cmath>
#include <cstring>
#endif

namespace nbk {
namespace i64 {

typedef unsigned long long u64;
typedef long long s64;

// a b 2^-64 or up to 3 less, for a, b <= 2^63: the product of the low halves
// is left out, and below 2^63 the cross products cannot carry out.
NB_HD u64 mulhi(u64 a, u64 b)
{
    const unsigned ah = (unsigned)(a >> 32), al = (unsigned)a, bh = (unsigned)(b >> 32), bl = (unsigned)b;
    const u64 t = (u64)ah * bl + (u64)al * bh;
    return (u64)ah * bh + (t >> 32);
}

NB_HD u64 bits_of(double x)
{
#ifdef __CUDA_ARCH__
    return (u64)__double_as_longlong(x);
#else
    u64 b;
    memcpy(&b, &x, 8);
    return b;
#endif
}

NB_HD double of_bits(u64 b)
{
#ifdef __CUDA_ARCH__
    return __longlong_as_double((s64)b);
#else
    double x;
    memcpy(&x, &b, 8);
    return x;
#endif
}

NB_HD int clz32(unsigned x)
{
#ifdef __CUDA_ARCH__
    return __clz((int)x);
#else
    return x ? __builtin_clz(x) : 32;
#endif
}
NB_HD int clz64(u64 x)
{
    const unsigned hi = (unsigned)(x >> 32);
    return clz32(hi ? hi : (unsigned)x) + (hi ? 0 : 32);
}

NB_HD int imin(int a, int b) { return a < b ? a : b; }
NB_HD int imax(int a, int b) { return a > b ? a : b; }

// +-m 2^(e - 62) with bit 62 of m the highest one set, or m = 0.
struct Num {
    u64 m;
    int e;
    bool neg;
};
constexpr int kZeroExp = -128;   // exponent kept for a value that is 0
// Byte k of w as a signed number: exponents in range fit one.
NB_HD int signed_byte(unsigned w, int k) { return (int)(w << (24 - 8 * k)) >> 24; }

// The values that this arithmetic takes: 0 and 2^-100 <= |x| < 2^100 (a
// difference of two such values that is not 0 is at least 2^-152, and no
// factor over- or underflows).
NB_HD bool in_range(double x)
{
    const u64 b = bits_of(x) & 0x7fffffffffffffffULL;
    return b == 0 || (b >> 52) - 923 < 200;
}
NB_HD bool eps2_in_range(double eps2) { return eps2 > 0.0 && in_range(eps2); }

// x = m 2^(e - 61) for x in range.
struct Fix {
    s64 m;
    int e;
};
NB_HD Fix to_fix(double x)
{
    const u64 b = bits_of(x);
    const int f = (int)((b >> 52) & 0x7ff);
    const s64 m = (s64)(((b << 9) & 0x1ffffffffffffe00ULL) | 0x2000000000000000ULL);
    Fix r;
    r.m = f == 0 ? 0 : ((s64)b < 0 ? -m : m);
    r.e = f == 0 ? kZeroExp : f - 1023;
    return r;
}
NB_HD Num to_num(double x)
{
    const Fix f = to_fix(x);
    Num r;
    r.m = (u64)(f.m < 0 ? -f.m : f.m) << 1;
    r.e = f.e;
    r.neg = f.m < 0;
    return r;
}

// a - b: as a Num, with what lies below 2^-61 of the larger one cut off (a
// difference that cancels is exact), and rounded to nearest FP64.
NB_HD Num diff(const Fix &a, const Fix &b, double &x)
{
    const int E = imax(a.e, b.e);
    const s64 d = (a.m >> imin(E - a.e, 63)) - (b.m >> imin(E - b.e, 63));
    const u64 n = (u64)(d < 0 ? -d : d);
    const int lz = clz64(n) - 1;
    Num r;
    r.neg = d < 0;
    r.m = n << (lz & 63);
    r.e = n == 0 ? -1022 : E + 1 - lz;
    x = of_bits((((u64)(unsigned)(r.e + 1022) << 52) + (r.m >> 10) + ((r.m >> 9) & 1)) |
                ((u64)d & 0x8000000000000000ULL));
    return r;
}

// +-m 2^s rounded to nearest FP64.
NB_HD double pack(u64 m, int lz, int s, bool neg)
{
    const u64 n = m << (lz & 63);
    const u64 b = ((u64)(unsigned)(1023 + 62 - lz + s) << 52) + (n >> 11) + ((n >> 10) & 1);
    return of_bits(neg ? b | 0x8000000000000000ULL : b);
}

// eps^2 = m 2^(e - 60) with e even, 2^60 <= m < 2^62.
struct Eps {
    u64 m;
    int e;
};
NB_HD Eps make_eps(double eps2)
{
    const Num n = to_num(eps2);
    Eps r;
    r.e = n.e - (n.e & 1);
    r.m = n.m >> (2 - (n.e & 1));
    return r;
}

// 1/sqrt in single precision, relative error below 2^-22.
NB_HD float rsqrt_seed(float f)
{
#ifdef __CUDA_ARCH__
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(f));
    return y;
#else
    return (float)(1.0 / std::sqrt((double)f));
#endif
}

// 1/r = Y 2^(-63 - h) with r^2 = |x|^2 + eps^2.
NB_HD u64 inv_dist(const Num x[3], const Eps &eps, int &h)
{
    // r^2 = S 2^(E - 59), four terms below 2^61 each
    const int E = imax(imax(2 * x[0].e, 2 * x[1].e), imax(2 * x[2].e, eps.e));
    const u64 S = (mulhi(x[0].m, x[0].m) >> imin(1 + E - 2 * x[0].e, 63)) +
                  (mulhi(x[1].m, x[1].m) >> imin(1 + E - 2 * x[1].e, 63)) +
                  (mulhi(x[2].m, x[2].m) >> imin(1 + E - 2 * x[2].e, 63)) + (eps.m >> imin(1 + E - eps.e, 63));
    // = f 2^(2 h), F = f 2^61 in [2^61, 2^63): E is even and S at least 2^59
    const bool low = S < (1ULL << 61);
    const u64 F = low ? S << 2 : S;
    h = (E >> 1) + (low ? 0 : 1);
    // y0 = Yi 2^-24 from the SFU, pulled below 1, then y0 (1 + e/2 + 3/8 e^2)
    // with e = 1 - f y0^2 (below 2^-20; the next term is below 2^-62)
    const unsigned Yi = (unsigned)(rsqrt_seed((float)(unsigned)(F >> 31)) * 0x1.fffffcp38f);
    const s64 e = (s64)((1ULL << 60) - mulhi(F, ((u64)Yi * Yi) << 15));   // in 2^-60
    const int e10 = (int)(e >> 10);
    const s64 c = (e >> 1) + ((((s64)e10 * e10) >> 40) * 3 >> 3);
    return ((u64)Yi << 39) + (u64)(((s64)Yi * c) >> 21);   // 1/sqrt(f) in 2^-63
}

// m / r.
NB_HD double pair_potential(const Num x[3], const Num &m, const Eps &eps)
{
    int h;
    const u64 H = mulhi(m.m, inv_dist(x, eps, h)) << 1;
    const double mr = pack(H, clz32((unsigned)(H >> 32)), m.e - 62 - h, m.neg);
    return m.m == 0 ? 0.0 : mr;
}

// m / r, m / r^3 and b = -3 (x . u) / r^2 with r^2 = |x|^2 + eps^2.
NB_HD void pair_factors(const Num x[3], const Num u[3], const Num &m, const Eps &eps, double &mr, double &mr3,
                        double &b)
{
    int h;
    const u64 Y = inv_dist(x, eps, h);
    const u64 Z = mulhi(Y, Y) << 1;   // 1/f in 2^-63, r^2 = f 2^(2 h)
    const u64 H = mulhi(m.m, Y) << 1, T = mulhi(H, Z);
    mr = pack(H, clz32((unsigned)(H >> 32)), m.e - 62 - h, m.neg);
    mr3 = pack(T, clz32((unsigned)(T >> 32)), m.e - 61 - 3 * h, m.neg);
    mr = m.m == 0 ? 0.0 : mr;
    mr3 = m.m == 0 ? 0.0 : mr3;
    // x . u = t 2^(G - 59), three terms below 2^61
    const int g0 = x[0].e + u[0].e, g1 = x[1].e + u[1].e, g2 = x[2].e + u[2].e, G = imax(imax(g0, g1), g2);
    const s64 a0 = (s64)(mulhi(x[0].m, u[0].m) >> imin(1 + G - g0, 63));
    const s64 a1 = (s64)(mulhi(x[1].m, u[1].m) >> imin(1 + G - g1, 63));
    const s64 a2 = (s64)(mulhi(x[2].m, u[2].m) >> imin(1 + G - g2, 63));
    const s64 t = (x[0].neg != u[0].neg ? -a0 : a0) + (x[1].neg != u[1].neg ? -a1 : a1) +
                  (x[2].neg != u[2].neg ? -a2 : a2);
    const u64 B = mulhi((u64)(t < 0 ? -t : t), Z) * 3;
    b = pack(B, clz64(B), G - 58 - 2 * h, t >= 0);
    b = B == 0 ? 0.0 : b;
}

}  // namespace i64
}  // namespace nbk
