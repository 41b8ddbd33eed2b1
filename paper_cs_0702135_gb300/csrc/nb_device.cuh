// nb_device.cuh -- device arithmetic shared by every kernel that predicts,
// corrects or sums pair forces, so that the single-system step, the ensemble
// step and the reverse mode evaluate the same formulas bit for bit.
#pragma once

#include <cuda_runtime.h>

#include <cfloat>

#include "nb_internal.cuh"

namespace nbk {
namespace dev {

constexpr double kTick = 0x1p-40;  // one tick in N-body time units

// The GB300's FP64 pipe serves an SM one warp instruction in 20 clocks, a warp
// one in 66 however many lanes are active and however independent they are,
// and conversions between integers, FP32 and FP64 are such instructions too
// (measured; a division or square root takes ~600 clocks).  What is only a
// move of bits is therefore done on the integer pipe, without branches: a
// function that works on a range of exponents sets `bad` outside it, and the
// caller redoes the whole expression with the FP64 operations once at its end
// (written volatile, or in a function of its own, so that the compiler does
// not evaluate them ahead of that test).
__device__ __forceinline__ double mul_volatile(double x, double y)
{
    double r;
    asm volatile("mul.rn.f64 %0, %1, %2;" : "=d"(r) : "d"(x), "d"(y));
    return r;
}

// d 2^-40, rounded to nearest.  Up to 2^52 ticks the integer goes into the
// significand of 2^12, whose last place is 2^-40, and 2^12 is subtracted: exact.
__device__ __forceinline__ double ticks_to_time(long long d)
{
    if ((unsigned long long)d < (1ULL << 52))
        return __dsub_rn(__longlong_as_double(d | 0x40B0000000000000LL), 4096.0);
    double r;
    asm volatile("cvt.rn.f64.s64 %0, %1;" : "=d"(r) : "l"(d));
    return mul_volatile(r, kTick);
}

// 2^e as FP64, -1022 <= e <= 1023.
__device__ __forceinline__ double pow2d(int e) { return __hiloint2double((1023 + e) << 20, 0); }

// Whether x's exponent lies in [2^(lo), 2^(lo + n)) (not zero, not finite: no).
template <int LO, int N>
__device__ __forceinline__ bool exponent_in(double x)
{
    return ((unsigned)__double2hiint(x) & 0x7fffffffu) - ((unsigned)(1023 + LO) << 20) < ((unsigned)N << 20);
}

// x 2^e, |e| <= 130, by moving the exponent field (exact).
__device__ __forceinline__ double scale2(double x, int e, bool &bad)
{
    bad = bad || !exponent_in<-823, 1600>(x);
    return __hiloint2double(__double2hiint(x) + (e << 20), __double2loint(x));
}

// dt / 2 for dt >= 0 from ticks_to_time.
__device__ __forceinline__ double half_dt(double dt)
{
    const int hi = __double2hiint(dt);
    return __hiloint2double(hi != 0 ? hi - (1 << 20) : 0, __double2loint(dt));
}

// 1/sqrt(x) on the SFU: the PTX approximate reciprocal square root with
// flush-to-zero (one MUFU instruction; relative error about 2^-23).  r^2 >=
// eps^2 is never subnormal, so the denormal handling of rsqrtf() would only
// cost issue slots here.
__device__ __forceinline__ float rsqrt_sfu(float x)
{
    float y;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Knuth's TwoSum: hi + lo absorbs x, with the rounding error of hi + x in lo.
__device__ __forceinline__ void two_sum_acc(float &hi, float &lo, float x)
{
    float s = hi + x;
    float bb = s - hi;
    float e = (hi - (s - bb)) + (x - bb);
    hi = s;
    lo += e;
}

// Sum of two double-single values (h, l) += (h2, l2).
__device__ __forceinline__ void ds_add(float &h, float &l, float h2, float l2)
{
    float s = h + h2;
    float bb = s - h;
    float e = (h - (s - bb)) + (h2 - bb);
    h = s;
    l = (l + l2) + e;
}

// Lane l ends up holding, for value index e = l >> (5 - log2 P), the DS sum of
// value e over all 32 lanes; P is a power of two <= 32.
template <int P>
__device__ __forceinline__ void warp_reduce_scatter(float (&h)[P], float (&lo)[P], int lane)
{
    int c = P;
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) {
        if (c > 1) {
            const bool up = (lane & off) != 0;
            const int half = c / 2;
#pragma unroll
            for (int k = 0; k < P / 2; ++k) {
                if (k < half) {
                    const float sh = up ? h[k] : h[k + half], sl = up ? lo[k] : lo[k + half];
                    float kh = up ? h[k + half] : h[k], kl = up ? lo[k + half] : lo[k];
                    const float rh = __shfl_xor_sync(0xffffffffu, sh, off);
                    const float rl = __shfl_xor_sync(0xffffffffu, sl, off);
                    ds_add(kh, kl, rh, rl);
                    h[k] = kh;
                    lo[k] = kl;
                }
            }
            c = half;
        } else {
            const float rh = __shfl_xor_sync(0xffffffffu, h[0], off);
            const float rl = __shfl_xor_sync(0xffffffffu, lo[0], off);
            ds_add(h[0], lo[0], rh, rl);
        }
    }
}

// a / C rounded to nearest, for the constants C = 3, 12, 20 of the predictor
// and corrector, without an FP64 division (a long sequence on the GB300's
// narrow FP64 pipe): q0 = RN(a y) with y = RN(1/C) is within one ulp of a/C
// (1/C is rounded with relative error 2^-54 for these C), the residual
// r = a - C q0 is exact in one FMA, and RN(q0 + r y) is then RN(a/C) by
// Markstein's theorem (IBM J. Res. Dev. 34, 1990).  Operands outside
// 2^-900 < |a| < 2^1000 (zero with its sign, huge, not finite) take the plain
// division; the range test reads the exponent bits on the integer pipe.
template <int C>
__device__ __forceinline__ double div_core(double a)
{
    static_assert(C == 3 || C == 12 || C == 20, "reciprocal error checked for 3, 12, 20 only");
    constexpr double y = 1.0 / C;
    const double q0 = __dmul_rn(a, y);
    const double r = __fma_rn(-q0, (double)C, a);
    return __fma_rn(r, y, q0);
}

template <int C>
__device__ __forceinline__ double div_by(double a)
{
    const unsigned hi = (unsigned)__double2hiint(a) & 0x7FFFFFFFu;
    if (hi >= (123u << 20) && hi < (2023u << 20)) return div_core<C>(a);
    return __ddiv_rn(a, (double)C);
}

// The same without the branch: `bad` outside the range.
template <int C>
__device__ __forceinline__ double div_by(double a, bool &bad)
{
    bad = bad || !exponent_in<123 - 1023, 1900>(a);
    return div_core<C>(a);
}

// Hermite predictor (Section 2), round-to-nearest in the formula's order:
//   x_p = x + (v + (dt/2)(a + (dt/3) k)) dt,   v_p = v + (a + (dt/2) k) dt.
// dt/2 is taken as dt * 0.5, the same number (halving is exact for every dt on
// the tick grid), which saves an FP64 division on the GB300's small FP64 pipe.
// With h = dt/2 and q = dt/3 given (one division per particle, not per axis):
__device__ __forceinline__ void predict1hq(double x, double v, double a, double k, double dt,
                                           double h, double q, double &xp, double &vp)
{
    xp = __dadd_rn(x, __dmul_rn(__dadd_rn(v, __dmul_rn(h, __dadd_rn(a, __dmul_rn(q, k)))), dt));
    vp = __dadd_rn(v, __dmul_rn(__dadd_rn(a, __dmul_rn(h, k)), dt));
}

__device__ __forceinline__ void predict1(double x, double v, double a, double k, double dt,
                                         double &xp, double &vp)
{
    predict1hq(x, v, a, k, dt, __dmul_rn(dt, 0.5), div_by<3>(dt), xp, vp);
}

// State loads: plain, or past L1 (CG) for state that other SMs may have
// written earlier in the same launch.
template <bool CG, typename T>
__device__ __forceinline__ T ldst(const T *p)
{
    if (CG) return __ldcg(p);
    return *p;
}

// All three axes of particle i of `s` (component-major, stride n).
template <bool CG = false>
__device__ __forceinline__ void predict3(const State &s, long long i, long long n, double dt,
                                         double xp[3], double vp[3])
{
    // a time step needs no range test: 0 (exact) or 2^-40 .. 2^22
    const double h = half_dt(dt), q = div_core<3>(dt);
#pragma unroll
    for (int c = 0; c < 3; ++c)
        predict1hq(ldst<CG>(&s.x[c * n + i]), ldst<CG>(&s.v[c * n + i]), ldst<CG>(&s.a[c * n + i]),
                   ldst<CG>(&s.k[c * n + i]), dt, h, q, xp[c], vp[c]);
}

// A predicted FP64 position split into double-single: x = hi + lo to 2^-48.
__device__ __forceinline__ void split_ds(double x, float &hi, float &lo)
{
    hi = __double2float_rn(x);
    lo = __double2float_rn(__dsub_rn(x, (double)hi));
}

// RN32(x) and RN32(x - RN32(x)) on the integer pipe (~15 instructions; a split
// by conversions is four FP64 instructions).  x = (-1)^s M 2^(e-1075): the top
// 24 bits of M round half to even by the remainder R of the low 29, and the
// rest R (- 2^29 if rounded up) is an integer of at most 29 bits, converted to
// FP32 (rounded to nearest) and scaled exactly.  `bad` outside [2^-70, 2^120).
__device__ __forceinline__ void split_ds_int(double x, float &hi, float &lo, bool &bad)
{
    bad = bad || !exponent_in<-70, 190>(x);
    const unsigned xh = (unsigned)__double2hiint(x), xl = (unsigned)__double2loint(x);
    const unsigned e = (xh >> 20) & 0x7ffu;
    const unsigned t = ((xh & 0x7fffffffu) - (896u << 20)) << 3 | xl >> 29;   // truncated to FP32
    const unsigned R = xl & 0x1fffffffu;
    const bool up = R + (t & 1u) > 0x10000000u;
    hi = __uint_as_float((t + up) | (xh & 0x80000000u));
    int r = (int)R - (up ? 0x20000000 : 0);
    r = (int)xh < 0 ? -r : r;
    lo = __int2float_rn(r) * __uint_as_float((e - (1075u - 127u)) << 23);
}
__device__ __forceinline__ float to_float_int(double x, bool &bad)
{
    bad = bad || !exponent_in<-70, 190>(x);
    const unsigned xh = (unsigned)__double2hiint(x), xl = (unsigned)__double2loint(x);
    const unsigned t = ((xh & 0x7fffffffu) - (896u << 20)) << 3 | xl >> 29;
    return __uint_as_float((t + ((xl & 0x1fffffffu) + (t & 1u) > 0x10000000u)) | (xh & 0x80000000u));
}
__device__ __forceinline__ float to_float_volatile(double x)
{
    float y;
    asm volatile("cvt.rn.f32.f64 %0, %1;" : "=f"(y) : "d"(x));
    return y;
}
// RN32(x) for an x that is bad: a zero (a system in a plane, a particle at rest) is
// still a move of bits.
__device__ __forceinline__ bool is_zero(double x) { return (__double_as_longlong(x) << 1) == 0; }
__device__ __forceinline__ float to_float_rest(double x)
{
    return is_zero(x) ? __int_as_float(__double2hiint(x)) : to_float_volatile(x);
}
__device__ __forceinline__ float to_float_int(double x)
{
    bool bad = false;
    const float y = to_float_int(x, bad);
    return bad ? to_float_rest(x) : y;
}
// A position's two words and a velocity where at least one of them was bad: what is
// in range stays.
__device__ __forceinline__ void split_rest(double x, double v, float &hi, float &lo, float &u)
{
    if (!exponent_in<-70, 190>(x)) {
        hi = to_float_rest(x);
        lo = is_zero(x) ? 0.0f : to_float_volatile(__dsub_rn(x, (double)hi));
    }
    if (!exponent_in<-70, 190>(v)) u = to_float_rest(v);
}

// A position split into double-single and a velocity in FP32, all axes.
__device__ __forceinline__ void split_record(const double x[3], const double v[3], float hi[3], float lo[3],
                                             float u[3])
{
    bool bad = false;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        split_ds_int(x[c], hi[c], lo[c], bad);
        u[c] = to_float_int(v[c], bad);
    }
    if (bad)
#pragma unroll
        for (int c = 0; c < 3; ++c) split_rest(x[c], v[c], hi[c], lo[c], u[c]);
}

__device__ __forceinline__ double norm3(double u0, double u1, double u2)
{
    return __dsqrt_rn(__dadd_rn(__dadd_rn(__dmul_rn(u0, u0), __dmul_rn(u1, u1)), __dmul_rn(u2, u2)));
}

// Block level of a raw step: k of the largest 2^-k <= dt_raw, from the FP64
// exponent field (dt_raw >= 2^-40 is a normal number), clamped to k >= kmin.
// Returns false when dt_raw is not a number or below 2^-40.
__device__ __forceinline__ bool level_of(double dt_raw, int kmin, int &level)
{
    if (isnan(dt_raw) || dt_raw < 0x1p-40) return false;
    int k;
    if (isinf(dt_raw)) {
        k = kmin;
    } else {
        const long long bits = __double_as_longlong(dt_raw);
        k = 1023 - (int)((bits >> 52) & 0x7FF);
        if (k < kmin) k = kmin;
    }
    level = k;
    return true;
}

// Halve at once; double by one level only when the new time is a multiple of
// the doubled step; never above the largest step.
__device__ __forceinline__ int next_level(int k_old, int k_q, long long t_new, int kmin)
{
    if (k_q > k_old) return k_q;
    if (k_q < k_old && k_old > kmin) {
        const long long twice_old = 1LL << (kTickBits - k_old + 1);
        if ((t_new & (twice_old - 1)) == 0) return k_old - 1;
    }
    return k_old;
}

// Start-up step eta_init |a| / |k|; +infinity when the jerk vanishes.
__device__ __forceinline__ double initial_dt(const double a[3], const double k[3], double eta_init)
{
    const double nk = norm3(k[0], k[1], k[2]);
    return nk == 0.0 ? (double)INFINITY : __ddiv_rn(__dmul_rn(eta_init, norm3(a[0], a[1], a[2])), nk);
}

// Level of the Aarseth step
//   dt_raw = sqrt(eta (|a| |s| + |k|^2) / (|k| |c| + |s|^2))
// from FP32 values of the four squared norms, where they decide it: dt_raw's
// binade is that of the FP32 estimate R of dt_raw^2 unless R lies within 2^-12
// of a power of four, and the estimate's error, with conversions, three-term
// sums, approximate square roots and the division, is below 2^-18.  False (the
// caller evaluates the FP64 formulas) there, and where a norm or R is outside
// the range in which FP32 keeps its precision (zero and non-finite included).
// A square root or division in FP64 takes ~600 clocks, this ~100.
__device__ __forceinline__ float sqrt_sfu(float x)
{
    float y;
    asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
__device__ __forceinline__ bool level_estimate(float na2, float nk2, float ns2, float nc2, float eta, int kmin,
                                               int &level)
{
    const float lo = fminf(fminf(na2, nk2), fminf(ns2, nc2)), hi = fmaxf(fmaxf(na2, nk2), fmaxf(ns2, nc2));
    const float num = fmaf(sqrt_sfu(na2), sqrt_sfu(ns2), nk2);
    const float den = fmaf(sqrt_sfu(nk2), sqrt_sfu(nc2), ns2);
    const float R = __fdividef(eta * num, den);
    if (!(lo >= 0x1p-100f && hi <= 0x1p110f && R >= 0x1p-72f && R <= 0x1p60f) ||
        !(na2 == na2 && nk2 == nk2 && ns2 == ns2 && nc2 == nc2))
        return false;
    const int b = __float_as_int(R), e = (b >> 23) - 127, m = b & 0x7fffff;
    if ((e & 1) ? m >= 0x800000 - 0x800 : m < 0x800) return false;
    level = max(-(e >> 1), kmin);
    return true;
}

// The corrector's arithmetic for one axis when the step is a power of two,
// dt = 2^e (every block step): multiplications by powers of two move the
// exponent (scale2), dt/3 is the rounded third with its exponent moved, and
// the other operations are those of correct_axis_any in its order, so the
// results are the same bits with 24 FP64 operations instead of ~47.
struct AxisStep {
    double x, v, s1, c;   // new position and velocity; s1 and crackle of the step criterion
};
__device__ __forceinline__ AxisStep correct_axis(double x, double v, double a, double k, double ap, double kp,
                                                 int e, bool &bad)
{
    AxisStep r;
    const double d = __dsub_rn(a, ap);
    const double a3 = __dadd_rn(scale2(d, 1, bad), scale2(__dadd_rn(k, kp), e, bad));
    const double a2 = __dsub_rn(__dmul_rn(-3.0, d), scale2(__dadd_rn(scale2(k, 1, bad), kp), e, bad));
    const double w = __dadd_rn(a, scale2(__dmul_rn(1.0 / 3.0, k), e, bad));
    const double xp = __dadd_rn(x, scale2(__dadd_rn(v, scale2(w, e - 1, bad)), e, bad));
    const double vp = __dadd_rn(v, scale2(__dadd_rn(a, scale2(k, e - 1, bad)), e, bad));
    const double a2_3 = div_by<3>(a2, bad);   // a2 / 12 is a quarter of it
    r.x = __dadd_rn(xp, scale2(__dadd_rn(scale2(a2_3, -2, bad), div_by<20>(a3, bad)), 2 * e, bad));
    r.v = __dadd_rn(vp, scale2(__dadd_rn(a2_3, scale2(a3, -2, bad)), e, bad));
    r.c = scale2(__dmul_rn(6.0, a3), -3 * e, bad);
    r.s1 = __dadd_rn(scale2(a2, 1 - 2 * e, bad), scale2(r.c, e, bad));
    return r;
}

// The same for any step and any values.
__device__ __forceinline__ AxisStep correct_axis_any(double x, double v, double a, double k, double ap, double kp,
                                                  long long ticks)
{
    AxisStep r;
    const double dt = ticks_to_time(ticks);
    const double h = __dmul_rn(dt, 0.5), q3 = div_by<3>(dt);
    const double dt2 = __dmul_rn(dt, dt);
    const double dt3 = __dmul_rn(dt2, dt);
    double xp, vp;
    predict1hq(x, v, a, k, dt, h, q3, xp, vp);
    const double d = __dsub_rn(a, ap);
    const double a3 = __dadd_rn(__dmul_rn(2.0, d), __dmul_rn(__dadd_rn(k, kp), dt));
    const double a2 = __dsub_rn(__dmul_rn(-3.0, d), __dmul_rn(__dadd_rn(__dmul_rn(2.0, k), kp), dt));
    r.x = __dadd_rn(xp, __dmul_rn(__dadd_rn(div_by<12>(a2), div_by<20>(a3)), dt2));
    // a3 / 4 as a3 * 0.25: the same real number, so the same rounded result
    r.v = __dadd_rn(vp, __dmul_rn(__dadd_rn(div_by<3>(a2), __dmul_rn(a3, 0.25)), dt));
    const double s0 = __ddiv_rn(__dmul_rn(2.0, a2), dt2);
    r.c = __ddiv_rn(__dmul_rn(6.0, a3), dt3);
    r.s1 = __dadd_rn(s0, __dmul_rn(r.c, dt));
    return r;
}

// Where correct_axis was bad: an axis at rest (a system in a plane) moves nothing, the
// sums of its zeros being +0; else the general form.  128 bodies in a plane, graph
// run: 27.7 us a step, 32.9 with the general form after the other, 31.7 with it alone.
static __device__ __noinline__ AxisStep correct_axis_rest(double x, double v, double a, double k, double ap, double kp,
                                                      long long ticks)
{
    const long long any = __double_as_longlong(v) | __double_as_longlong(a) | __double_as_longlong(k) |
                          __double_as_longlong(ap) | __double_as_longlong(kp);
    if (any == 0 && ticks > 0) return {is_zero(x) ? 0.0 : x, 0.0, 0.0, 0.0};
    return correct_axis_any(x, v, a, k, ap, kp, ticks);
}

// e of a step of `ticks` = 2^(e + 40) ticks; false for any other step.
__device__ __forceinline__ bool step_exponent(long long ticks, int &e)
{
    e = 63 - kTickBits - __clzll(ticks);
    return ticks > 0 && (ticks & (ticks - 1)) == 0 && e >= -kTickBits && e <= 0;
}

// The Aarseth step's level from the FP64 norms (false: below 2^-40).
static __device__ __noinline__ bool level_exact(double na, double nk, double ns, double nc, double eta, int kmin,
                                            int &level)
{
    const double num = __dadd_rn(__dmul_rn(na, ns), __dmul_rn(nk, nk));
    const double den = __dadd_rn(__dmul_rn(nk, nc), __dmul_rn(ns, ns));
    const double dt_raw = den == 0.0 ? (double)INFINITY : __dsqrt_rn(__ddiv_rn(__dmul_rn(eta, num), den));
    return level_of(dt_raw, kmin, level);
}

__device__ __forceinline__ float norm2_f(float x, float y, float z) { return fmaf(x, x, fmaf(y, y, z * z)); }

// Hermite corrector and Aarseth step for particle i of `s` (Section 2).  In
// the paper's notation a, k are the old values (in s) and a_p, k_p the new:
//   a3 = 2 (a - a_p) + (k + k_p) dt,   a2 = -3 (a - a_p) - (2 k + k_p) dt,
//   x = x_p + (a2/12 + a3/20) dt^2,    v = v_p + (a2/3 + a3/4) dt.
// Snap s0 = 2 a2 / dt^2, crackle c = 6 a3 / dt^3, s1 = s0 + c dt, and
//   dt_new = sqrt(eta (|a_p| |s1| + |k_p|^2) / (|k_p| |c| + |s1|^2)),
// quantised by level_of and next_level (level_fixed > 0 keeps that level).
// x_p, v_p are recomputed with predict1, bit for bit the values the force
// saw.  Returns false when the new step fell below 2^-40.
template <bool CG = false>
__device__ __forceinline__ bool correct_particle(const State &s, long long i, long long stride,
                                                 long long tn, const double ap[3], const double kp[3],
                                                 double eta, int level_min, int level_fixed)
{
    const long long ticks = tn - ldst<CG>(&s.t[i]);
    double s1[3], cr[3];
    int ex;
    const bool block_step = step_exponent(ticks, ex);
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const long long e = c * stride + i;
        const double x = ldst<CG>(&s.x[e]), v = ldst<CG>(&s.v[e]), a = ldst<CG>(&s.a[e]),
                     k = ldst<CG>(&s.k[e]);
        bool bad = !block_step;
        AxisStep r = correct_axis(x, v, a, k, ap[c], kp[c], ex, bad);
        if (bad) r = correct_axis_rest(x, v, a, k, ap[c], kp[c], ticks);
        s.x[e] = r.x;
        s.v[e] = r.v;
        s.a[e] = ap[c];
        s.k[e] = kp[c];
        s1[c] = r.s1;
        cr[c] = r.c;
    }
    s.t[i] = tn;
    if (level_fixed > 0) {
        s.lev[i] = level_fixed;
        return true;
    }
    float f[4][3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        f[0][c] = to_float_int(ap[c]);
        f[1][c] = to_float_int(kp[c]);
        f[2][c] = to_float_int(s1[c]);
        f[3][c] = to_float_int(cr[c]);
    }
    int kq;
    bool ok = true;
    if (!level_estimate(norm2_f(f[0][0], f[0][1], f[0][2]), norm2_f(f[1][0], f[1][1], f[1][2]),
                        norm2_f(f[2][0], f[2][1], f[2][2]), norm2_f(f[3][0], f[3][1], f[3][2]),
                        to_float_int(eta), level_min, kq)) {
        ok = level_exact(norm3(ap[0], ap[1], ap[2]), norm3(kp[0], kp[1], kp[2]), norm3(s1[0], s1[1], s1[2]),
                         norm3(cr[0], cr[1], cr[2]), eta, level_min, kq);
        if (!ok) kq = kTickBits;
    }
    s.lev[i] = next_level(ldst<CG>(&s.lev[i]), kq, tn, level_min);
    return ok;
}

// ---------------------------------------------------------------------------
// Single-precision mirror of the FP64 state, for j records predicted with FP32
// Taylor increments: position as double-single (x_hi + mass, x_lo), velocity,
// acceleration and jerk in FP32, as five float4 arrays of the particle count.
struct Mirror {
    float4 *h, *l, *v, *a, *k;
};

// The mirror of particle i from its FP64 state (component-major, stride n).
template <bool CG = false>
__device__ __forceinline__ void write_mirror(const State &s, const Mirror &mr, long long i, long long n)
{
    double x[3], v[3];
    float hi[3], lo[3], u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) x[c] = ldst<CG>(&s.x[c * n + i]), v[c] = ldst<CG>(&s.v[c * n + i]);
    split_record(x, v, hi, lo, u);
    mr.h[i] = make_float4(hi[0], hi[1], hi[2], to_float_int(ldst<CG>(&s.m[i])));
    mr.l[i] = make_float4(lo[0], lo[1], lo[2], 0.0f);
    mr.v[i] = make_float4(u[0], u[1], u[2], 0.0f);
    mr.a[i] = make_float4(to_float_int(ldst<CG>(&s.a[i])), to_float_int(ldst<CG>(&s.a[n + i])),
                          to_float_int(ldst<CG>(&s.a[2 * n + i])), 0.0f);
    mr.k[i] = make_float4(to_float_int(ldst<CG>(&s.k[i])), to_float_int(ldst<CG>(&s.k[n + i])),
                          to_float_int(ldst<CG>(&s.k[2 * n + i])), 0.0f);
}

// (hi, lo) + d in double-single: TwoSum of hi and d, then renormalised.
__device__ __forceinline__ void ds_add_f(float hi, float lo, float d, float &ho, float &lout)
{
    const float s = hi + d;
    const float bb = s - hi;
    const float e = (hi - (s - bb)) + (d - bb);
    const float l2 = lo + e;
    ho = s + l2;
    lout = l2 - (ho - s);
}

// j record of particle i, dt ticks after its own time, from the mirror: the
// predictor's Taylor increments (Section 2) in FP32,
//   dx = (v + (dt/2)(a + (dt/3) k)) dt,   v_p = v + (a + (dt/2) k) dt,
// and the position accumulated in double-single, x_p = (x_hi + x_lo) + dx.
template <bool CG = false>
__device__ __forceinline__ void predict_j32(const Mirror &mr, long long i, long long dt_ticks,
                                            float4 &ph, float4 &pl, float4 &pv)
{
    const float dt = (float)dt_ticks * 0x1p-40f;
    const float h = 0.5f * dt, q = dt * (1.0f / 3.0f);
    const float4 xh = ldst<CG>(&mr.h[i]), xl = ldst<CG>(&mr.l[i]), v = ldst<CG>(&mr.v[i]),
                 a = ldst<CG>(&mr.a[i]), k = ldst<CG>(&mr.k[i]);
    ds_add_f(xh.x, xl.x, fmaf(h, fmaf(q, k.x, a.x), v.x) * dt, ph.x, pl.x);
    ds_add_f(xh.y, xl.y, fmaf(h, fmaf(q, k.y, a.y), v.y) * dt, ph.y, pl.y);
    ds_add_f(xh.z, xl.z, fmaf(h, fmaf(q, k.z, a.z), v.z) * dt, ph.z, pl.z);
    pv.x = fmaf(fmaf(h, k.x, a.x), dt, v.x);
    pv.y = fmaf(fmaf(h, k.y, a.y), dt, v.y);
    pv.z = fmaf(fmaf(h, k.z, a.z), dt, v.z);
    ph.w = xh.w;
    pl.w = 0.0f;
    pv.w = 0.0f;
}

// correct_particle spread over the four lanes of a quad (lanes 4u .. 4u+3 of
// a warp), for blocks too small to fill the GPU: the corrector is a chain of
// FP64 operations, and on the GB300 an FP64 warp instruction occupies the SM's
// narrow FP64 pipe for many cycles however few of its lanes are active, so
// one particle's three axes on three lanes issue a third of the one-thread
// form's FP64 instructions.  Each lane
// evaluates exactly the operations of correct_particle for its axis, in the
// same order, so the results are the same bits.
//
// Every lane of the warp must call this together (it shuffles over the whole
// warp).  Lane q = lane & 3 of a quad passes component q of the new
// acceleration and jerk (lane 3: any finite value, e.g. that of axis 2) and
// the same particle i as its quad; `active` false (the whole quad) computes
// on a valid i without storing.  Returns false (on every lane of an active
// quad) when the new step fell below 2^-40.
template <bool CG = false>
__device__ __forceinline__ bool correct_particle_quad(const State &s, long long i, long long stride,
                                                      long long tn, double apc, double kpc,
                                                      double eta, int level_min, int level_fixed,
                                                      bool active)
{
    const int lane = threadIdx.x & 31, q = lane & 3, base = lane & ~3;
    const int c = q < 3 ? q : 2;          // lane 3 shadows axis 2 without storing
    const bool own = active && q < 3;
    const long long ticks = tn - ldst<CG>(&s.t[i]);
    const long long e = c * stride + i;
    const double x = ldst<CG>(&s.x[e]), v = ldst<CG>(&s.v[e]), a = ldst<CG>(&s.a[e]),
                 k = ldst<CG>(&s.k[e]);
    const int lev_old = ldst<CG>(&s.lev[i]);
    int ex;
    bool bad = !step_exponent(ticks, ex);
    AxisStep r = correct_axis(x, v, a, k, apc, kpc, ex, bad);
    if (bad) r = correct_axis_rest(x, v, a, k, apc, kpc, ticks);
    // every lane of the quad has read the old state before any lane stores
    __syncwarp();
    if (own) {
        s.x[e] = r.x;
        s.v[e] = r.v;
        s.a[e] = apc;
        s.k[e] = kpc;
    }
    if (level_fixed > 0) {
        if (active && q == 0) {
            s.t[i] = tn;
            s.lev[i] = level_fixed;
        }
        return true;
    }
    // squared norms of a_p, k_p, s1, c on every lane of the quad: lane 3
    // shadows axis 2 and adds nothing
    float n2[4] = {to_float_int(apc), to_float_int(kpc), to_float_int(r.s1), to_float_int(r.c)};
#pragma unroll
    for (int w = 0; w < 4; ++w) {
        n2[w] = q < 3 ? n2[w] * n2[w] : 0.0f;
        n2[w] += __shfl_xor_sync(0xffffffffu, n2[w], 1);
        n2[w] += __shfl_xor_sync(0xffffffffu, n2[w], 2);
    }
    int kq = 0;
    bool ok = true;
    const bool known = level_estimate(n2[0], n2[1], n2[2], n2[3], to_float_int(eta), level_min, kq);
    if (__any_sync(0xffffffffu, active && !known)) {
        // |a_p|, |k_p|, |s1|, |c| on lanes 0..3 of the quad, each as norm3 forms it
        const double sq0 = __dmul_rn(apc, apc), sq1 = __dmul_rn(kpc, kpc);
        const double sq2 = __dmul_rn(r.s1, r.s1), sq3 = __dmul_rn(r.c, r.c);
        double w[3];
#pragma unroll
        for (int cc = 0; cc < 3; ++cc) {
            const double t0 = __shfl_sync(0xffffffffu, sq0, base + cc);
            const double t1 = __shfl_sync(0xffffffffu, sq1, base + cc);
            const double t2 = __shfl_sync(0xffffffffu, sq2, base + cc);
            const double t3 = __shfl_sync(0xffffffffu, sq3, base + cc);
            w[cc] = q == 0 ? t0 : (q == 1 ? t1 : (q == 2 ? t2 : t3));
        }
        const double nrm = __dsqrt_rn(__dadd_rn(__dadd_rn(w[0], w[1]), w[2]));
        const double na = __shfl_sync(0xffffffffu, nrm, base + 0);
        const double nk = __shfl_sync(0xffffffffu, nrm, base + 1);
        const double ns = __shfl_sync(0xffffffffu, nrm, base + 2);
        const double nc = __shfl_sync(0xffffffffu, nrm, base + 3);
        if (!known) {
            ok = level_exact(na, nk, ns, nc, eta, level_min, kq);
            if (!ok) kq = kTickBits;
        }
    }
    if (active && q == 0) {
        s.t[i] = tn;
        s.lev[i] = next_level(lev_old, kq, tn, level_min);
    }
    return ok;
}

// FP32 pair terms of Eq. 1 (attractive sign; pair terms of the Appendix A
// kernel) from the separation dx = x_j - x_i and the velocity difference
// u = v_j - v_i.  SOFT = false drops pairs at r = 0; GUARD drops the pair
// j == i.
template <bool SOFT, bool GUARD>
__device__ __forceinline__ void pair_terms(float dx, float dy, float dz, float ux, float uy, float uz,
                                           float m, float eps2, float acc[3], float jk[3], float &pot,
                                           int j, int i)
{
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
    const float rv = fmaf(dx, ux, fmaf(dy, uy, dz * uz));
    float rinv = rsqrt_sfu(r2);
    if (!SOFT) rinv = (r2 > 0.0f) ? rinv : 0.0f;
    if (GUARD) rinv = (j == i) ? 0.0f : rinv;
    const float rinv2 = rinv * rinv;
    const float mr = m * rinv;             // m_j / r
    const float mr3 = mr * rinv2;          // m_j / r^3
    const float b = -3.0f * rv * rinv2;    // -3 (dx . dv) / r^2
    acc[0] = fmaf(mr3, dx, acc[0]);
    acc[1] = fmaf(mr3, dy, acc[1]);
    acc[2] = fmaf(mr3, dz, acc[2]);
    const float qx = fmaf(b, dx, ux);
    const float qy = fmaf(b, dy, uy);
    const float qz = fmaf(b, dz, uz);
    jk[0] = fmaf(mr3, qx, jk[0]);
    jk[1] = fmaf(mr3, qy, jk[1]);
    jk[2] = fmaf(mr3, qz, jk[2]);
    pot -= mr;
}

// One FP32 pair interaction on double-single positions, dx = x_j - x_i formed
// as (x_j,hi - x_i,hi) + (x_j,lo - x_i,lo).
template <bool SOFT, bool GUARD>
__device__ __forceinline__ void pair_ds(const float4 &p, const float4 &l, const float4 &w,
                                        const float xh[3], const float xl[3], const float vi[3],
                                        float eps2, float acc[3], float jk[3], float &pot,
                                        int j = 0, int i = 1)
{
    const float dx = (p.x - xh[0]) + (l.x - xl[0]);
    const float dy = (p.y - xh[1]) + (l.y - xl[1]);
    const float dz = (p.z - xh[2]) + (l.z - xl[2]);
    pair_terms<SOFT, GUARD>(dx, dy, dz, w.x - vi[0], w.y - vi[1], w.z - vi[2], p.w, eps2, acc, jk, pot,
                            j, i);
}

// The i side of a pair in the packed form below: the x and y components
// negated and paired, z kept as it is.
struct IDS {
    float2 nh, nl, nv;   // (-x_hi, -y_hi), (-x_lo, -y_lo), (-v_x, -v_y)
    float zh, zl, vz;
};

__device__ __forceinline__ IDS make_ids(const float4 &p, const float4 &l, const float4 &v)
{
    IDS I;
    I.nh = make_float2(-p.x, -p.y);
    I.nl = make_float2(-l.x, -l.y);
    I.nv = make_float2(-v.x, -v.y);
    I.zh = p.z; I.zl = l.z; I.vz = v.z;
    return I;
}

// pair_ds with the x and y components of the three differences taken by
// packed two-lane FP32 adds (add.f32x2): four instructions instead of eight,
// each lane rounded exactly as the scalar subtraction it replaces
// (RN(a + (-b)) = RN(a - b)), so the result is bit for bit that of pair_ds.
// The FMA pipe does the same work; the saving is issue slots.
template <bool SOFT, bool GUARD>
__device__ __forceinline__ void pair_ds_packed(const float4 &p, const float4 &l, const float4 &w,
                                               const IDS &I, float eps2, float acc[3], float jk[3],
                                               float &pot, int j = 0, int i = 1)
{
    const float2 dh = __fadd2_rn(make_float2(p.x, p.y), I.nh);
    const float2 dl = __fadd2_rn(make_float2(l.x, l.y), I.nl);
    const float2 d = __fadd2_rn(dh, dl);
    const float2 u = __fadd2_rn(make_float2(w.x, w.y), I.nv);
    const float dz = (p.z - I.zh) + (l.z - I.zl);
    pair_terms<SOFT, GUARD>(d.x, d.y, dz, u.x, u.y, w.z - I.vz, p.w, eps2, acc, jk, pot, j, i);
}

// Block size of a force launch: read on the device when the host does not know it.
__device__ __forceinline__ int read_na(const ForceArgs &fa)
{
    return fa.na_dev ? *fa.na_dev : fa.na_host;
}

// Index loads of padding lanes are clamped into [0, n).
__device__ __forceinline__ int clamp_index(int i, int n) { return min(max(i, 0), n - 1); }

// One particle's acc, jerk, pot into the public output layout.
__device__ __forceinline__ void store_result(const ForceOut &o, int a, const double r[kComp])
{
    if (o.acc) {
        o.acc[3 * (long long)a + 0] = r[0];
        o.acc[3 * (long long)a + 1] = r[1];
        o.acc[3 * (long long)a + 2] = r[2];
    }
    if (o.jerk) {
        o.jerk[3 * (long long)a + 0] = r[3];
        o.jerk[3 * (long long)a + 1] = r[4];
        o.jerk[3 * (long long)a + 2] = r[5];
    }
    if (o.pot) o.pot[a] = r[6];
}

// Component c (0-2 acc, 3-5 jerk, 6 pot) of output a.
__device__ __forceinline__ void write_combined(const ForceOut &o, int c, int a, double s)
{
    if (c < 3) {
        if (o.acc) o.acc[3 * (long long)a + c] = s;
    } else if (c < 6) {
        if (o.jerk) o.jerk[3 * (long long)a + (c - 3)] = s;
    } else if (o.pot) {
        o.pot[a] = s;
    }
}

// ---------------------------------------------------------------------------
// Summation variants (Section 6): single-precision pair terms with IEEE
// round-to-nearest operations in a fixed order, and the exact integer
// arithmetic of the GRAPE-style fixed-point sums.

// The seven single-precision terms of j on i, each scaled as stated above;
// false when r2 = 0 (the terms are then not numbers and must be skipped).
__device__ __forceinline__ bool pair_rn(const float4 &p, const float4 &l, const float4 &w,
                                        const float xh[3], const float xl[3], const float vi[3],
                                        float eps2, float sa, float sk, float sp, float t[7])
{
    const float dx0 = __fadd_rn(__fsub_rn(p.x, xh[0]), __fsub_rn(l.x, xl[0]));
    const float dx1 = __fadd_rn(__fsub_rn(p.y, xh[1]), __fsub_rn(l.y, xl[1]));
    const float dx2 = __fadd_rn(__fsub_rn(p.z, xh[2]), __fsub_rn(l.z, xl[2]));
    const float u0 = __fsub_rn(w.x, vi[0]);
    const float u1 = __fsub_rn(w.y, vi[1]);
    const float u2 = __fsub_rn(w.z, vi[2]);
    const float d2 = __fadd_rn(__fadd_rn(__fmul_rn(dx0, dx0), __fmul_rn(dx1, dx1)), __fmul_rn(dx2, dx2));
    const float r2 = __fadd_rn(d2, eps2);
    const float rv = __fadd_rn(__fadd_rn(__fmul_rn(dx0, u0), __fmul_rn(dx1, u1)), __fmul_rn(dx2, u2));
    const float rinv = __frcp_rn(__fsqrt_rn(r2));
    const float rinv2 = __fmul_rn(rinv, rinv);
    const float mr = __fmul_rn(p.w, rinv);
    const float mr3 = __fmul_rn(mr, rinv2);
    const float b = __fmul_rn(__fmul_rn(-3.0f, rv), rinv2);
    const float fa = __fmul_rn(mr3, sa), fk = __fmul_rn(mr3, sk), fp = __fmul_rn(mr, sp);
    t[0] = __fmul_rn(fa, dx0);
    t[1] = __fmul_rn(fa, dx1);
    t[2] = __fmul_rn(fa, dx2);
    t[3] = __fmul_rn(fk, __fadd_rn(u0, __fmul_rn(b, dx0)));
    t[4] = __fmul_rn(fk, __fadd_rn(u1, __fmul_rn(b, dx1)));
    t[5] = __fmul_rn(fk, __fadd_rn(u2, __fmul_rn(b, dx2)));
    t[6] = -fp;
    return r2 != 0.0f;
}

// Two-lane arithmetic for two pairs at once.  A packed product that feeds a packed
// sum comes out as one multiply-add even where both carry .rn (the results of the
// intrinsics and of add.rn/mul.rn.f32x2 differ from the scalar operations'), so
// such a product (mul2s) is a packed multiply-add of -0, which rounds the product
// itself and cannot be contracted; the -0 comes from constant memory, where it is
// not known at compile time.
static __constant__ float2 c_neg_zero2 = {-0.0f, -0.0f};

__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 mul2s(float2 a, float2 b) { return __ffma2_rn(a, b, c_neg_zero2); }

// True where inv_sqrt_fast2 below does not give RN(1 / RN(sqrt(x))): x outside
// [2^-87, 2^126], or within 6 ulps below a power of four (a square root whose
// significand is all ones is the exception of Markstein's theorem).
__device__ __forceinline__ bool inv_sqrt_hard(float x)
{
    const unsigned b = __float_as_uint(x);
    return b - 0x14000000u > 0x6A800000u || ((b + 0x800006u) & 0xffffffu) < 6u;
}

// RN(1 / RN(sqrt(x))) for two x that are not inv_sqrt_hard, from the SFU's
// approximate y ~ 1/sqrt(x) (relative error about 2^-22.9) by the final steps
// of Markstein (IBM J. Res. Dev. 34, 1990): with s0 = x y and the exact
// residual x - s0^2, s = RN(s0 + (x - s0^2) y/2) is the rounded square root;
// y1 = RN(y + (1 - s y) y) is within an ulp of its reciprocal and, with the
// exact residual 1 - s y1, RN(y1 + (1 - s y1) y1) is the rounded reciprocal.
// Compared on the GB300 with __frcp_rn(__fsqrt_rn(x)) for every non-negative
// single-precision x (tests/test_gpu_arith.py): the same bits wherever
// inv_sqrt_hard is false.  Two x share every operation here: the index-order sums
// of 1820 active on 65536 bodies took 583 us with the intrinsics, 502 with this
// form and packed pairs.
__device__ __forceinline__ float2 inv_sqrt_fast2(float2 x)
{
    const float2 y = make_float2(rsqrt_sfu(x.x), rsqrt_sfu(x.y));
    const float2 s0 = mul2(x, y);
    const float2 s = fma2(fma2(neg2(s0), s0, x), mul2(y, f2(0.5f)), s0);
    const float2 y1 = fma2(fma2(neg2(s), y, f2(1.0f)), y, y);
    return fma2(fma2(neg2(s), y1, f2(1.0f)), y1, y1);
}

__device__ __forceinline__ float2 inv_sqrt_rn2(float2 x)
{
    float2 r = inv_sqrt_fast2(x);
    if (inv_sqrt_hard(x.x) || inv_sqrt_hard(x.y)) {
        r.x = __frcp_rn(__fsqrt_rn(x.x));
        r.y = __frcp_rn(__fsqrt_rn(x.y));
    }
    return r;
}

// RN(sqrt(x)) for two x by the first of those steps.
__device__ __forceinline__ float2 sqrt_rn2(float2 x)
{
    const float2 y = make_float2(rsqrt_sfu(x.x), rsqrt_sfu(x.y));
    const float2 s0 = mul2(x, y);
    float2 s = fma2(fma2(neg2(s0), s0, x), mul2(y, f2(0.5f)), s0);
    if (inv_sqrt_hard(x.x) || inv_sqrt_hard(x.y)) {
        s.x = __fsqrt_rn(x.x);
        s.y = __fsqrt_rn(x.y);
    }
    return s;
}

// One side of two pairs: hi and lo position words, velocity (of the i side
// negated), mass.
struct Side2 {
    float2 h[3], l[3], v[3], m;
};

// pair_rn on two pairs: j of each lane (J), i of each lane negated (N).  Every
// operation is pair_rn's, in its order, rounded per lane, so the bits are the
// same.  UNIT: the scale factors are 1 and their multiplications are left out
// (exact).  Returns r2 (a lane with r2 = 0 holds no numbers in t).
template <bool UNIT>
__device__ __forceinline__ float2 pair_rn2(const Side2 &J, const Side2 &N, float eps2, float sa, float sk,
                                           float sp, float2 t[7])
{
    float2 dx[3], u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        dx[c] = add2(add2(J.h[c], N.h[c]), add2(J.l[c], N.l[c]));
        u[c] = add2(J.v[c], N.v[c]);
    }
    const float2 d2 = add2(add2(mul2s(dx[0], dx[0]), mul2s(dx[1], dx[1])), mul2s(dx[2], dx[2]));
    const float2 r2 = add2(d2, f2(eps2));
    const float2 rv = add2(add2(mul2s(dx[0], u[0]), mul2s(dx[1], u[1])), mul2s(dx[2], u[2]));
    const float2 rinv = inv_sqrt_rn2(r2);
    const float2 rinv2 = mul2(rinv, rinv);
    const float2 mr = mul2(J.m, rinv);
    const float2 mr3 = mul2(mr, rinv2);
    const float2 b = mul2(mul2(f2(-3.0f), rv), rinv2);
    const float2 fa = UNIT ? mr3 : mul2(mr3, f2(sa)), fk = UNIT ? mr3 : mul2(mr3, f2(sk));
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const float2 q = add2(u[c], mul2s(b, dx[c]));
        // scaled terms go on into packed sums (split_add2)
        t[c] = UNIT ? mul2(fa, dx[c]) : mul2s(fa, dx[c]);
        t[3 + c] = UNIT ? mul2(fk, q) : mul2s(fk, q);
    }
    t[6] = UNIT ? neg2(mr) : mul2s(mr, f2(-sp));
    return r2;
}

// The sort keys of two pairs, min(mr3 sqrt(d2), FLT_MAX) with pair_rn's operations;
// r2 in rr (a pair with r2 = 0 has no key).
__device__ __forceinline__ float2 pair_key2(const Side2 &J, const Side2 &N, float eps2, float2 &rr)
{
    float2 dx[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) dx[c] = add2(add2(J.h[c], N.h[c]), add2(J.l[c], N.l[c]));
    const float2 d2 = add2(add2(mul2s(dx[0], dx[0]), mul2s(dx[1], dx[1])), mul2s(dx[2], dx[2]));
    rr = add2(d2, f2(eps2));
    const float2 rinv = inv_sqrt_rn2(rr);
    const float2 key = mul2(mul2(mul2(J.m, rinv), mul2(rinv, rinv)), sqrt_rn2(d2));
    return make_float2(fminf(key.x, FLT_MAX), fminf(key.y, FLT_MAX));
}

// The records of two particles side by side, and one in both lanes negated.
__device__ __forceinline__ Side2 side2(const float4 &p0, const float4 &l0, const float4 &v0,
                                       const float4 &p1, const float4 &l1, const float4 &v1)
{
    Side2 s;
    s.h[0] = make_float2(p0.x, p1.x), s.h[1] = make_float2(p0.y, p1.y), s.h[2] = make_float2(p0.z, p1.z);
    s.l[0] = make_float2(l0.x, l1.x), s.l[1] = make_float2(l0.y, l1.y), s.l[2] = make_float2(l0.z, l1.z);
    s.v[0] = make_float2(v0.x, v1.x), s.v[1] = make_float2(v0.y, v1.y), s.v[2] = make_float2(v0.z, v1.z);
    s.m = make_float2(p0.w, p1.w);
    return s;
}
__device__ __forceinline__ Side2 side2_neg(const float4 &p, const float4 &l, const float4 &v)
{
    Side2 s = side2(p, l, v, p, l, v);
#pragma unroll
    for (int c = 0; c < 3; ++c) s.h[c] = neg2(s.h[c]), s.l[c] = neg2(s.l[c]), s.v[c] = neg2(s.v[c]);
    return s;
}

__device__ __forceinline__ void load_i(const JDS &J, int i, float xh[3], float xl[3], float vi[3])
{
    const float4 p = J.pos_hi[i], l = J.pos_lo[i], v = J.vel[i];
    xh[0] = p.x; xh[1] = p.y; xh[2] = p.z;
    xl[0] = l.x; xl[1] = l.y; xl[2] = l.z;
    vi[0] = v.x; vi[1] = v.y; vi[2] = v.z;
}

// ---------------------------------------------------------------------------
// Fixed point

struct Scale {
    float sc[3];    // 2^s: acc, jerk, pot
    double inv[3];  // 2^-s
};

__device__ __forceinline__ int exp_above(unsigned bits)
{
    const int be = (int)((bits >> 23) & 0xFF);
    return be == 0 ? -126 : be - 126;
}

__device__ __forceinline__ int floor_half(int a) { return a >= 0 ? a / 2 : -((1 - a) / 2); }

// Scales from the bounds.  With eps2 >= 2^F, every mass < 2^Em and every
// |vx| + |vy| + |vz| < 2^Ev (Em, Ev at least -64), the terms obey
//   |acc| <= mj / r^2 < 2^(Em - F),   |pot| = mj / r < 2^(Em - floor(F/2)),
//   |jerk| <= 4 mj |dv| / r^3 < 2^(3 + Em + Ev - floor(3F/2))
// up to single-precision rounding, which the factor 2 between 2^56 and 2^57
// absorbs; s = min(56 - e, 126).  False when eps2 is not a normal float or a
// scale falls below -126.
__device__ __forceinline__ bool fixed_scale(const unsigned *bounds, float eps2, Scale &S)
{
    const int be = (int)((__float_as_uint(eps2) >> 23) & 0xFF);
    if (be == 0 || be == 255) return false;
    const int F = be - 127;
    const int Em = max(exp_above(bounds[0]), -64), Ev = max(exp_above(bounds[1]), -64);
    const int e[3] = {Em - F, 3 + Em + Ev - floor_half(3 * F), Em - floor_half(F)};
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const int s = min(56 - e[q], 126);
        if (s < -126) return false;
        S.sc[q] = __int_as_float((s + 127) << 23);
        S.inv[q] = __longlong_as_double((long long)(1023 - s) << 52);
    }
    return true;
}

// Exact integer rounding of a term |t| < 2^57 - 2^34 on the FP32 pipe.  For
// C = 1.5 * 2^(23+g), s = fl(t + C) stays in C's binade while |t| < 2^(22+g),
// so s - C is t rounded to a multiple of 2^g and bits(s) - bits(C) is that
// multiple's count.  With g = 35, 13 and 0:
//   s1 = fl(t + C1),  r  = t - (s1 - C1)      |r|  <= 2^34, exact
//   s2 = fl(r + C2),  r2 = r - (s2 - C2)      |r2| <= 2^12, exact
//   s3 = fl(r2 + C3)                          r2 rounded half to even
// and round_half_even(t) = a1 2^35 + a2 2^13 + a3 with a_k = bits(s_k) -
// bits(C_k) (the first two parts are even, so the tie rule carries over).  A
// tile adds the raw bit patterns in 32 bits (mod 2^32) and subtracts the
// constants once: the true sums stay below 2^28 in magnitude.
constexpr float kC1 = 0x1.8p58f, kC2 = 0x1.8p36f, kC3 = 0x1.8p23f;

__device__ __forceinline__ void split_add(float t, unsigned &a1, unsigned &a2, unsigned &a3)
{
    const float s1 = __fadd_rn(t, kC1);
    const float r = __fsub_rn(t, __fsub_rn(s1, kC1));
    const float s2 = __fadd_rn(r, kC2);
    const float r2 = __fsub_rn(r, __fsub_rn(s2, kC2));
    const float s3 = __fadd_rn(r2, kC3);
    a1 += __float_as_uint(s1);
    a2 += __float_as_uint(s2);
    a3 += __float_as_uint(s3);
}

// split_add on two terms: the same roundings per lane, C - s taken as the
// exact multiply-add s (-1) + C; the terms must not be plain packed products
// (see mul2s).
__device__ __forceinline__ void split_add2(float2 t, unsigned &a1, unsigned &a2, unsigned &a3)
{
    const float2 s1 = add2(t, f2(kC1));
    const float2 r = add2(t, fma2(s1, f2(-1.0f), f2(kC1)));
    const float2 s2 = add2(r, f2(kC2));
    const float2 r2 = add2(r, fma2(s2, f2(-1.0f), f2(kC2)));
    const float2 s3 = add2(r2, f2(kC3));
    a1 += __float_as_uint(s1.x) + __float_as_uint(s1.y);
    a2 += __float_as_uint(s2.x) + __float_as_uint(s2.y);
    a3 += __float_as_uint(s3.x) + __float_as_uint(s3.y);
}

// The integer sum of a tile of `cnt` split terms.
__device__ __forceinline__ long long tile_sum(unsigned a1, unsigned a2, unsigned a3, unsigned cnt)
{
    const int q1 = (int)(a1 - cnt * __float_as_uint(kC1));
    const int q2 = (int)(a2 - cnt * __float_as_uint(kC2));
    const int q3 = (int)(a3 - cnt * __float_as_uint(kC3));
    return ((long long)q1 << 35) + ((long long)q2 << 13) + (long long)q3;
}

// (hi, lo) += x, a 128-bit two's-complement sum.
__device__ __forceinline__ void add128(long long &hi, unsigned long long &lo, long long x)
{
    const unsigned long long l2 = lo + (unsigned long long)x;
    hi += (x >> 63) + (l2 < lo ? 1 : 0);
    lo = l2;
}

// |Y| = H 2^64 + L  ->  fl64(fl64(H) 2^64 + fl64(L)), with Y's sign.
__device__ __forceinline__ double i128_to_double(long long hi, unsigned long long lo)
{
    const bool neg = hi < 0;
    if (neg) {
        lo = ~lo + 1ULL;
        hi = ~hi + (lo == 0ULL ? 1 : 0);
    }
    const double d = __dadd_rn(__dmul_rn(__ull2double_rn((unsigned long long)hi), 0x1p64),
                               __ull2double_rn(lo));
    return neg ? -d : d;
}

}  // namespace dev
}  // namespace nbk
