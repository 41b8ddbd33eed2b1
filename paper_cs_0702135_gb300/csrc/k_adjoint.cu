// k_adjoint.cu -- reverse-mode kernels: the vector-Jacobian product of the
// direct-summation force, and the transposes of the (linear) Hermite
// corrector and predictor for a fixed shared time step.  The paper has no
// gradients; these extend its method to a differentiable trajectory.
//
// Force VJP.  For every ordered pair (i, j), j != i, with d = x_j - x_i,
// w = v_j - v_i, r^2 = |d|^2 + eps^2, s = d.w and cotangents (abar_i, kbar_i)
// on acc_i and jerk_i, the derivatives of abar_i.acc_i + kbar_i.jerk_i are
//   g_d(abar, kbar) = m_j [ abar/r^3 - 3 (s kbar + (kbar.d) w)/r^5
//                           + (-3 (abar.d + kbar.w)/r^5 + 15 s (kbar.d)/r^7) d ]
//   g_w(kbar)       = m_j [ kbar/r^3 - 3 (kbar.d) d/r^5 ]
//   g_m             = abar.d/r^3 + kbar.(w/r^3 - 3 s d/r^5)        (w.r.t. m_j)
// with xbar_j += g_d, xbar_i -= g_d, vbar_j += g_w, vbar_i -= g_w.  Both g_d
// and g_w are even in (d, w) and linear in (abar, kbar), so for particle k
// the contributions as i (partner p as j, weight m_p) and as j (partner p as
// i, weight m_k) fold into one evaluation with
//   A = m_k abar_p - m_p abar_k,   K = m_k kbar_p - m_p kbar_k:
//   xbar_k += G(A, K),   vbar_k += H(K),
//   mbar_k += -(abar_p.d + kbar_p.w)/r^3 + 3 s (kbar_p.d)/r^5,
// with d = x_p - x_k.  One k-parallel sweep, no atomics; each thread owns
// kVKR particles k (one in the FP64 twin) and streams the partners through
// shared memory in tiles, like the forward i-parallel kernel (double-single
// positions, FP32 pair arithmetic, TwoSum-promoted tile partials).
#include "nb_device.cuh"

namespace nbk {
namespace {

using namespace dev;

constexpr int kVNT = 128;  // partners per tile; FP64: threads per CTA
constexpr int kVDsNT = 64; // DS: threads per CTA
constexpr int kVUnroll = 4;   // DS: partner unrolling

// One particle's VJP record: (predicted) position and velocity, mass and the
// cotangents of its acc and jerk, in the layout of the context's precision.
__device__ __forceinline__ void write_vjp_record(int i, const double x[3], const double v[3], double m,
                                 const double ab[3], const double kb[3], int precision,
                                 VjpRecDS rec, VjpRec64 rec64)
{
    if (precision == NB_FP64) {
        rec64.x[i] = make_double4_32a(x[0], x[1], x[2], m);
        rec64.v[i] = make_double4_32a(v[0], v[1], v[2], 0.0);
        rec64.ab[i] = make_double4_32a(ab[0], ab[1], ab[2], 0.0);
        rec64.kb[i] = make_double4_32a(kb[0], kb[1], kb[2], 0.0);
    } else {
        float hi[3], lo[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) split_ds(x[c], hi[c], lo[c]);
        rec.ph[i] = make_float4(hi[0], hi[1], hi[2], __double2float_rn(m));
        rec.pl[i] = make_float4(lo[0], lo[1], lo[2], 0.0f);
        rec.v[i] = make_float4(__double2float_rn(v[0]), __double2float_rn(v[1]),
                               __double2float_rn(v[2]), 0.0f);
        rec.ab[i] = make_float4(__double2float_rn(ab[0]), __double2float_rn(ab[1]),
                                __double2float_rn(ab[2]), 0.0f);
        rec.kb[i] = make_float4(__double2float_rn(kb[0]), __double2float_rn(kb[1]),
                                __double2float_rn(kb[2]), 0.0f);
    }
}


// The k side of a pair: the x and y components of position and velocity
// negated and paired for the packed differences (see pair_ds_packed).
struct VjpK {
    IDS q;
    float m, ab[3], kb[3];
};

// One (k, p) pair in FP32 on double-single positions; acc[0..2] xbar,
// acc[3..5] vbar, acc[6] mbar.
template <bool SOFT, bool GUARD>
__device__ __forceinline__ void vjp_pair_ds(const VjpRec &P, const VjpK &Kp, float eps2,
                                            float acc[7], int p = 0, int k = 1)
{
    const float2 dxy = __fadd2_rn(__fadd2_rn(make_float2(P.ph.x, P.ph.y), Kp.q.nh),
                                  __fadd2_rn(make_float2(P.pl.x, P.pl.y), Kp.q.nl));
    const float2 wxy = __fadd2_rn(make_float2(P.v.x, P.v.y), Kp.q.nv);
    const float dx = dxy.x, dy = dxy.y, dz = (P.ph.z - Kp.q.zh) + (P.pl.z - Kp.q.zl);
    const float wx = wxy.x, wy = wxy.y, wz = P.v.z - Kp.q.vz;
    const float r2 = fmaf(dx, dx, fmaf(dy, dy, fmaf(dz, dz, eps2)));
    float rinv = rsqrt_sfu(r2);
    if (!SOFT) rinv = (r2 > 0.0f) ? rinv : 0.0f;
    if (GUARD) rinv = (p == k) ? 0.0f : rinv;
    const float rinv2 = rinv * rinv;
    const float r3 = rinv * rinv2;
    const float r5 = r3 * rinv2;
    const float r7 = r5 * rinv2;
    const float s = fmaf(dx, wx, fmaf(dy, wy, dz * wz));
    const float mk = Kp.m, mp = P.ph.w;
    const float Ax = fmaf(mk, P.ab.x, -mp * Kp.ab[0]);
    const float Ay = fmaf(mk, P.ab.y, -mp * Kp.ab[1]);
    const float Az = fmaf(mk, P.ab.z, -mp * Kp.ab[2]);
    const float Kx = fmaf(mk, P.kb.x, -mp * Kp.kb[0]);
    const float Ky = fmaf(mk, P.kb.y, -mp * Kp.kb[1]);
    const float Kz = fmaf(mk, P.kb.z, -mp * Kp.kb[2]);
    const float Ad = fmaf(Ax, dx, fmaf(Ay, dy, Az * dz));
    const float Kd = fmaf(Kx, dx, fmaf(Ky, dy, Kz * dz));
    const float Kw = fmaf(Kx, wx, fmaf(Ky, wy, Kz * wz));
    const float t5 = -3.0f * r5;
    const float cd = fmaf(t5, Ad + Kw, 15.0f * s * Kd * r7);   // coefficient of d in G
    const float cs = t5 * s;                                    // coefficient of K in G
    const float cw = t5 * Kd;                                   // coefficient of w in G, of d in H
    acc[0] += fmaf(r3, Ax, fmaf(cs, Kx, fmaf(cw, wx, cd * dx)));
    acc[1] += fmaf(r3, Ay, fmaf(cs, Ky, fmaf(cw, wy, cd * dy)));
    acc[2] += fmaf(r3, Az, fmaf(cs, Kz, fmaf(cw, wz, cd * dz)));
    acc[3] += fmaf(r3, Kx, cw * dx);
    acc[4] += fmaf(r3, Ky, cw * dy);
    acc[5] += fmaf(r3, Kz, cw * dz);
    const float apd = fmaf(P.ab.x, dx, fmaf(P.ab.y, dy, P.ab.z * dz));
    const float kpw = fmaf(P.kb.x, wx, fmaf(P.kb.y, wy, P.kb.z * wz));
    const float kpd = fmaf(P.kb.x, dx, fmaf(P.kb.y, dy, P.kb.z * dz));
    acc[6] += fmaf(-r3, apd + kpw, 3.0f * s * kpd * r5);
}

// R particles k per thread, tiles of kVNT partners.
template <int R, bool SOFT>
__global__ void __launch_bounds__(kVDsNT) k_force_vjp_ds(VjpArgs va)
{
    constexpr int NT = kVDsNT;
    const Plan P = va.plan;
    __shared__ float4 s_ph[kVNT], s_pl[kVNT], s_v[kVNT], s_ab[kVNT], s_kb[kVNT];
    const float eps2 = (float)va.eps2;
    const int tid = threadIdx.x;
    for (int w = blockIdx.x; w < P.items; w += gridDim.x) {
        const int ib = w % P.n_iblk, sl = w / P.n_iblk;
        const int j0 = sl * P.jslice;
        const int j1 = min(va.n, j0 + P.jslice);
        int kk[R], k[R];
        VjpK K[R];
        float hi[R][7], lo[R][7];
#pragma unroll
        for (int r = 0; r < R; ++r) {
            kk[r] = ib * NT * R + r * NT + tid;
            k[r] = clamp_index(kk[r], va.n);
            const float4 ph = va.rec.ph[k[r]], ab = va.rec.ab[k[r]], kb = va.rec.kb[k[r]];
            K[r].q = make_ids(ph, va.rec.pl[k[r]], va.rec.v[k[r]]);
            K[r].m = ph.w;
            K[r].ab[0] = ab.x, K[r].ab[1] = ab.y, K[r].ab[2] = ab.z;
            K[r].kb[0] = kb.x, K[r].kb[1] = kb.y, K[r].kb[2] = kb.z;
#pragma unroll
            for (int c = 0; c < 7; ++c) hi[r][c] = lo[r][c] = 0.0f;
        }
        for (int jt = j0; jt < j1; jt += kVNT) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < kVNT / NT; ++u) {
                const int t = tid + u * NT, j = jt + t;
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
                s_ph[t] = j < j1 ? va.rec.ph[j] : z;
                s_pl[t] = j < j1 ? va.rec.pl[j] : z;
                s_v[t] = j < j1 ? va.rec.v[j] : z;
                s_ab[t] = j < j1 ? va.rec.ab[j] : z;
                s_kb[t] = j < j1 ? va.rec.kb[j] : z;
            }
            __syncthreads();
            float t[R][7];
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < 7; ++c) t[r][c] = 0.0f;
            bool mine = false;
#pragma unroll
            for (int r = 0; r < R; ++r) mine |= (unsigned)(k[r] - jt) < (unsigned)kVNT;
            if (__any_sync(0xffffffffu, mine)) {
                for (int jj = 0; jj < kVNT; ++jj) {
                    VjpRec Pq;
                    Pq.ph = s_ph[jj]; Pq.pl = s_pl[jj]; Pq.v = s_v[jj]; Pq.ab = s_ab[jj]; Pq.kb = s_kb[jj];
#pragma unroll
                    for (int r = 0; r < R; ++r) vjp_pair_ds<SOFT, true>(Pq, K[r], eps2, t[r], jt + jj, k[r]);
                }
            } else {
#pragma unroll (kVUnroll)
                for (int jj = 0; jj < kVNT; ++jj) {
                    VjpRec Pq;
                    Pq.ph = s_ph[jj]; Pq.pl = s_pl[jj]; Pq.v = s_v[jj]; Pq.ab = s_ab[jj]; Pq.kb = s_kb[jj];
#pragma unroll
                    for (int r = 0; r < R; ++r) vjp_pair_ds<SOFT, false>(Pq, K[r], eps2, t[r]);
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < 7; ++c) two_sum_acc(hi[r][c], lo[r][c], t[r][c]);
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            if (kk[r] >= va.n) continue;
            double res[7];
#pragma unroll
            for (int c = 0; c < 7; ++c) res[c] = (double)hi[r][c] + (double)lo[r][c];
            if (P.S == 1) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    va.xbar[3 * (long long)k[r] + c] = res[c];
                    va.vbar[3 * (long long)k[r] + c] = res[3 + c];
                }
                va.mbar[k[r]] = res[6];
            } else {
#pragma unroll
                for (int c = 0; c < 7; ++c) va.part[((long long)sl * 7 + c) * va.n + k[r]] = res[c];
            }
        }
    }
}

// The DS sweep's particles per thread and slices.  Up to kVOneMax particles one
// k per thread and slices of one tile: the sweep is then short of CTAs (4096:
// 59 us, two k a thread 66, and 70 with 128-thread CTAs and slices of two tiles;
// 1024: 15 against 23 us; at the line they meet, with the step's other kernel:
// 8192 234 and 236 us, 10240 361 and 360, 16384 871 and 825).  Above, two k per thread, each partner record
// read from shared memory serving two pairs, and slices that make about
// kVWaves waves of the resident CTAs, dealt out as CTAs end (65536: 12.4 ms,
// 12.9 ms with one k; one wave 14.8 ms, three 12.7 ms).
constexpr int kVOneMax = 8192, kVWaves = 8;

Plan plan_vjp_ds(int n, int slots, long long part_cap, int &R)
{
    Plan p{};
    R = n <= kVOneMax ? 1 : 2;
    p.n_iblk = cdiv(n, kVDsNT * R);
    const long long tiles = cdiv(n, kVNT);
    long long L = R == 1 ? 1 : cdiv(tiles * p.n_iblk, (long long)kVWaves * slots);
    while (L < tiles && cdiv(tiles, L) * (long long)kComp * n > part_cap) ++L;
    p.jslice = (int)(L * kVNT);
    p.S = cdiv(n, p.jslice);
    p.items = p.n_iblk * p.S;
    return p;
}

// FP64 twin, one k per thread, partners through shared memory.
template <bool SOFT>
__global__ void __launch_bounds__(kVNT) k_force_vjp_f64(VjpArgs va)
{
    const Plan P = va.plan;
    __shared__ double4_32a s_x[kVNT], s_v[kVNT], s_a[kVNT], s_k[kVNT];
    const double eps2 = va.eps2;
    const int tid = threadIdx.x;
    for (int w = blockIdx.x; w < P.items; w += gridDim.x) {
        const int ib = w % P.n_iblk, sl = w / P.n_iblk;
        const int j0 = sl * P.jslice;
        const int j1 = min(va.n, j0 + P.jslice);
        const int kk = ib * kVNT + tid;
        const int k = clamp_index(kk, va.n);
        const double4_32a Xk = va.rec64.x[k], Vk = va.rec64.v[k], Ak = va.rec64.ab[k],
                          Kk = va.rec64.kb[k];
        double acc[7] = {0., 0., 0., 0., 0., 0., 0.};
        for (int jt = j0; jt < j1; jt += kVNT) {
            __syncthreads();
            const int j = jt + tid;
            const double4_32a z = make_double4_32a(0., 0., 0., 0.);
            s_x[tid] = j < j1 ? va.rec64.x[j] : z;
            s_v[tid] = j < j1 ? va.rec64.v[j] : z;
            s_a[tid] = j < j1 ? va.rec64.ab[j] : z;
            s_k[tid] = j < j1 ? va.rec64.kb[j] : z;
            __syncthreads();
            for (int jj = 0; jj < kVNT; ++jj) {
                const double4_32a Xp = s_x[jj], Vp = s_v[jj], Ap = s_a[jj], Kp = s_k[jj];
                const double dx = Xp.x - Xk.x, dy = Xp.y - Xk.y, dz = Xp.z - Xk.z;
                const double wx = Vp.x - Vk.x, wy = Vp.y - Vk.y, wz = Vp.z - Vk.z;
                const double r2 = fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2)));
                double rinv = rsqrt(r2);
                if (!SOFT) rinv = (r2 > 0.0) ? rinv : 0.0;
                rinv = (jt + jj == k) ? 0.0 : rinv;
                const double rinv2 = rinv * rinv, r3 = rinv * rinv2, r5 = r3 * rinv2, r7 = r5 * rinv2;
                const double s = fma(dx, wx, fma(dy, wy, dz * wz));
                const double mk = Xk.w, mp = Xp.w;
                const double Ax = mk * Ap.x - mp * Ak.x, Ay = mk * Ap.y - mp * Ak.y, Az = mk * Ap.z - mp * Ak.z;
                const double Kx = mk * Kp.x - mp * Kk.x, Ky = mk * Kp.y - mp * Kk.y, Kz = mk * Kp.z - mp * Kk.z;
                const double Ad = Ax * dx + Ay * dy + Az * dz;
                const double Kd = Kx * dx + Ky * dy + Kz * dz;
                const double Kw = Kx * wx + Ky * wy + Kz * wz;
                const double cd = -3.0 * r5 * (Ad + Kw) + 15.0 * s * Kd * r7;
                const double cs = -3.0 * r5 * s, cw = -3.0 * r5 * Kd;
                acc[0] += r3 * Ax + cs * Kx + cw * wx + cd * dx;
                acc[1] += r3 * Ay + cs * Ky + cw * wy + cd * dy;
                acc[2] += r3 * Az + cs * Kz + cw * wz + cd * dz;
                acc[3] += r3 * Kx + cw * dx;
                acc[4] += r3 * Ky + cw * dy;
                acc[5] += r3 * Kz + cw * dz;
                const double apd = Ap.x * dx + Ap.y * dy + Ap.z * dz;
                const double kpw = Kp.x * wx + Kp.y * wy + Kp.z * wz;
                const double kpd = Kp.x * dx + Kp.y * dy + Kp.z * dz;
                acc[6] += -r3 * (apd + kpw) + 3.0 * s * kpd * r5;
            }
        }
        if (kk < va.n) {
            if (P.S == 1) {
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    va.xbar[3 * (long long)k + c] = acc[c];
                    va.vbar[3 * (long long)k + c] = acc[3 + c];
                }
                va.mbar[k] = acc[6];
            } else {
#pragma unroll
                for (int c = 0; c < 7; ++c) va.part[((long long)sl * 7 + c) * va.n + k] = acc[c];
            }
        }
    }
}

__global__ void k_vjp_combine(VjpArgs va, int S)
{
    const long long total = 7LL * va.n;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e / va.n), k = (int)(e % va.n);
        double s = 0.0;
        for (int q = 0; q < S; ++q) s += va.part[((long long)q * 7 + c) * va.n + k];
        if (c < 3) va.xbar[3 * (long long)k + c] = s;
        else if (c < 6) va.vbar[3 * (long long)k + (c - 3)] = s;
        else va.mbar[k] = s;
    }
}

// Backward step, first half: from the cotangents (xb, vb, ab, kb) of the state
// after a step that started at `st`, the cotangents of the new acc and jerk
// (through the corrector's D = a - a1, a3 and a2, and the new state's own
// acc and jerk) go into the force-VJP records, together with the predicted
// positions and velocities of the step; ab, kb become the corrector's part of
// the old acc and jerk cotangents.
//   a2b = xb dt^2/12 + vb dt/3,  a3b = xb dt^2/20 + vb dt/4,  Db = 2 a3b - 3 a2b
//   a1b = ab - Db,  k1b = kb + (a3b - a2b) dt,  ab <- Db,  kb <- (a3b - 2 a2b) dt
__global__ void k_adj_pre(State st, double dt, const double *xb, const double *vb, double *ab,
                          double *kb, int precision, VjpRecDS rec, VjpRec64 rec64)
{
    const int n = st.n;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double xp[3], vp[3], a1b[3], k1b[3];
        predict3(st, i, n, dt, xp, vp);
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long q = 3LL * i + c;
            const double a2b = div_by<12>(xb[q] * dt * dt) + div_by<3>(vb[q] * dt);
            const double a3b = div_by<20>(xb[q] * dt * dt) + vb[q] * dt * 0.25;
            const double Db = 2.0 * a3b - 3.0 * a2b;
            a1b[c] = ab[q] - Db;
            k1b[c] = kb[q] + (a3b - a2b) * dt;
            ab[q] = Db;
            kb[q] = (a3b - 2.0 * a2b) * dt;
        }
        write_vjp_record(i, xp, vp, st.m[i], a1b, k1b, precision, rec, rec64);
    }
}

// Backward step, second half: add the force VJP to the cotangents of the
// predicted state and take them through the predictor's transpose:
//   xp = x + v dt + a h dt + k q h dt,   vp = v + a dt + k h dt.
__global__ void k_adj_post(int n, double dt, double *xb, double *vb, double *ab, double *kb,
                           double *mb, const double *xg, const double *vg, const double *mg)
{
    const double h = dt / 2.0, q = dt / 3.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const long long e = 3LL * i + c;
            const double xpb = xb[e] + xg[e], vpb = vb[e] + vg[e];
            xb[e] = xpb;
            vb[e] = xpb * dt + vpb;
            ab[e] += xpb * h * dt + vpb * dt;
            kb[e] += xpb * q * h * dt + vpb * h * dt;
        }
        mb[i] += mg[i];
    }
}

// Records for a VJP at the un-predicted state (the initial force), and the
// final accumulation of its result.
__global__ void k_adj_initial_rec(State st, const double *ab, const double *kb, int precision,
                                  VjpRecDS rec, VjpRec64 rec64)
{
    const int n = st.n;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        double x[3], v[3], a[3], k[3];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            x[c] = st.x[c * n + i];
            v[c] = st.v[c * n + i];
            a[c] = ab[3LL * i + c];
            k[c] = kb[3LL * i + c];
        }
        write_vjp_record(i, x, v, st.m[i], a, k, precision, rec, rec64);
    }
}

__global__ void k_add3(int n, double *dst, const double *src, double *dst2, const double *src2,
                       double *dstm, const double *srcm)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            dst[3LL * i + c] += src[3LL * i + c];
            dst2[3LL * i + c] += src2[3LL * i + c];
        }
        dstm[i] += srcm[i];
    }
}

// Acceleration and jerk of a full sweep (public layout) into the SoA state.
__global__ void k_set_ak(State st, const double *acc, const double *jerk)
{
    const int n = st.n;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x)
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            st.a[c * n + i] = acc[3LL * i + c];
            st.k[c * n + i] = jerk[3LL * i + c];
        }
}

// ---------------------------------------------------------------------------
// Trajectories with a shared power-of-two step dt: every particle is active in
// every step and all are at one time, so the host knows each block and no
// scheduler runs.  A step is the force sweep and one kernel that adds its
// slices, corrects (or takes the force as it is, at the start), writes the new
// state where the caller wants it (and to a checkpoint), and predicts the next
// step's j records.  32 particles a CTA: a warp per force component adds the
// slices, then a warp per axis does the FP64 chain, because a warp has one
// FP64 instruction in flight whatever its lanes.  (The device-driven step's
// seven launches and the copies took 95 us a step at 4096 bodies beside a
// force of 38 us.)

constexpr int kShNT = 256, kShP = 32;

// Value c of particle a: the sum of its slices in order, or the result itself.
__device__ __forceinline__ double sum_slices(const double *part, int S, int c, long long nb, long long a)
{
    double s = 0.0;
#pragma unroll 8
    for (int q = 0; q < S; ++q) s += part[((long long)q * kComp + c) * nb + a];
    return s;
}

__global__ void __launch_bounds__(kShNT) k_shared_step(SharedStep q)
{
    __shared__ double s_f[6][kShP];
    __shared__ double s_r[6][kShP];   // predicted x, v
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = q.src.n, i = blockIdx.x * kShP + lane;
    if (q.mode != kShPredict && warp < 6 && i < n) {
        const double *out = warp < 3 ? q.out.acc : q.out.jerk;
        s_f[warp][lane] = q.S > 1 && i >= q.a0 ? sum_slices(q.part, q.S, warp, n - q.a0, i - q.a0)
                                               : out[3LL * i + warp % 3];
    }
    __syncthreads();
    const double dt = pow2d(-q.level);
    if (warp < 3 && i < n) {
        const long long e = (long long)warp * n + i;
        double x = q.src.x[e], v = q.src.v[e], a = q.src.a[e], k = q.src.k[e];
        if (q.mode != kShPredict) {
            const double ap = s_f[warp][lane], kp = s_f[3 + warp][lane];
            if (q.mode == kShCorrect) {
                bool bad = false;
                AxisStep r = correct_axis(x, v, a, k, ap, kp, -q.level, bad);
                if (bad) r = correct_axis_rest(x, v, a, k, ap, kp, 1LL << (kTickBits - q.level));
                x = r.x, v = r.v;
            }
            a = ap, k = kp;
            q.dst.x[e] = x, q.dst.v[e] = v, q.dst.a[e] = a, q.dst.k[e] = k;
            if (q.copy.x) q.copy.x[e] = x, q.copy.v[e] = v, q.copy.a[e] = a, q.copy.k[e] = k;
        }
        if (q.predict) predict1hq(x, v, a, k, dt, half_dt(dt), div_core<3>(dt), s_r[warp][lane], s_r[3 + warp][lane]);
    }
    if (!q.predict) return;
    __syncthreads();
    if (warp >= 3 || i >= n) return;
    const double m = q.src.m[i];
    if (q.precision == NB_FP64) {
        if (warp == 0) q.jf.pos[i] = make_double4_32a(s_r[0][lane], s_r[1][lane], s_r[2][lane], m);
        if (warp == 1) q.jf.vel[i] = make_double4_32a(s_r[3][lane], s_r[4][lane], s_r[5][lane], 0.0);
        return;
    }
    const double xp[3] = {s_r[0][lane], s_r[1][lane], s_r[2][lane]}, vp[3] = {s_r[3][lane], s_r[4][lane], s_r[5][lane]};
    float hi[3], lo[3], u[3];
    split_record(xp, vp, hi, lo, u);
    if (warp == 0) q.jds.pos_hi[i] = make_float4(hi[0], hi[1], hi[2], to_float_int(m));
    else if (warp == 1) q.jds.pos_lo[i] = make_float4(lo[0], lo[1], lo[2], 0.0f);
    else q.jds.vel[i] = make_float4(u[0], u[1], u[2], 0.0f);
}

// After the last of `steps` shared steps: particle times, the block list and
// the counters as the device-driven steps leave them.
__global__ void k_shared_done(State s, Ctrl *ctrl, int *act, long long steps, int level)
{
    const int n = s.n;
    const long long t = ctrl->t_now + steps * (1LL << (kTickBits - level));
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < n; i += gridDim.x * blockDim.x) {
        s.t[i] = t;
        act[i] = i;
    }
}
// Every particle at time t with the shared step.
__global__ void k_shared_times(State s, long long t, int level)
{
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < s.n; i += gridDim.x * blockDim.x) {
        s.t[i] = t;
        s.lev[i] = level;
    }
}
__global__ void k_shared_ctrl(Ctrl *ctrl, int n, long long steps, int level)
{
    ctrl->t_now += steps * (1LL << (kTickBits - level));
    ctrl->t_next = ctrl->t_now;
    ctrl->n_active = n;
    ctrl->steps += steps;
    ctrl->interactions += steps * (long long)n * (long long)(n - 1);
}

// The reverse pass between two force VJPs, fused the same way: the slices of
// the last VJP added; its second half (k_adj_post's formulas) or the final
// accumulation; then the first half of the step before it (k_adj_pre's
// formulas) or the record of the initial state, as the next VJP's records.
// Every operation is written out, so the results do not depend on which parts
// share a launch.
__global__ void __launch_bounds__(kShNT) k_adj_step(AdjStep q)
{
    __shared__ double s_g[7][kShP];
    __shared__ double s_r[12][kShP];   // x, v, and the cotangents of acc and jerk
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int n = q.st.n, i = blockIdx.x * kShP + lane;
    if ((q.post || q.add) && warp < 7 && i < n) {
        if (q.S > 1) s_g[warp][lane] = sum_slices(q.part, q.S, warp, n, i);
        else s_g[warp][lane] = warp < 3 ? q.xg[3LL * i + warp] : (warp < 6 ? q.vg[3LL * i + warp - 3] : q.mg[i]);
    }
    __syncthreads();
    const double dt = pow2d(-q.level), h = half_dt(dt), third = div_core<3>(dt);
    if (warp < 3 && i < n) {
        const long long e = 3LL * i + warp;
        double xb = q.xb[e], vb = q.vb[e], ab = q.ab[e], kb = q.kb[e];
        if (q.post) {
            //   xp = x + v dt + a h dt + k q h dt,   vp = v + a dt + k h dt
            const double xpb = __dadd_rn(xb, s_g[warp][lane]), vpb = __dadd_rn(vb, s_g[3 + warp][lane]);
            xb = xpb;
            vb = __fma_rn(xpb, dt, vpb);
            ab = __dadd_rn(ab, __fma_rn(xpb, __dmul_rn(h, dt), __dmul_rn(vpb, dt)));
            kb = __dadd_rn(kb, __fma_rn(__dmul_rn(xpb, third), __dmul_rn(h, dt), __dmul_rn(vpb, __dmul_rn(h, dt))));
        } else if (q.add) {
            xb = __dadd_rn(xb, s_g[warp][lane]);
            vb = __dadd_rn(vb, s_g[3 + warp][lane]);
        }
        if (q.pre != kAdjNone) {
            const long long c = (long long)warp * n + i;
            const double x = q.st.x[c], v = q.st.v[c];
            if (q.pre == kAdjPre) {
                //   a2b = xb dt^2/12 + vb dt/3,  a3b = xb dt^2/20 + vb dt/4,  Db = 2 a3b - 3 a2b
                const double xd = __dmul_rn(xb, __dmul_rn(dt, dt)), vd = __dmul_rn(vb, dt);
                const double a2b = __dadd_rn(div_by<12>(xd), div_by<3>(vd));
                const double a3b = __dadd_rn(div_by<20>(xd), __dmul_rn(vd, 0.25));
                const double Db = __fma_rn(-3.0, a2b, __dmul_rn(2.0, a3b));
                s_r[6 + warp][lane] = __dsub_rn(ab, Db);
                s_r[9 + warp][lane] = __fma_rn(__dsub_rn(a3b, a2b), dt, kb);
                ab = Db;
                kb = __dmul_rn(__fma_rn(-2.0, a2b, a3b), dt);
                predict1hq(x, v, q.st.a[c], q.st.k[c], dt, h, third, s_r[warp][lane], s_r[3 + warp][lane]);
            } else {
                s_r[warp][lane] = x;
                s_r[3 + warp][lane] = v;
                s_r[6 + warp][lane] = ab;
                s_r[9 + warp][lane] = kb;
            }
        }
        q.xb[e] = xb, q.vb[e] = vb, q.ab[e] = ab, q.kb[e] = kb;
    }
    if (warp == 3 && i < n && (q.post || q.add)) q.mb[i] = __dadd_rn(q.mb[i], s_g[6][lane]);
    if (q.pre == kAdjNone) return;
    __syncthreads();
    // four warps share the record: position, velocity, two cotangents
    if (warp >= 4 || i >= n) return;
    const double r[3] = {s_r[3 * warp][lane], s_r[3 * warp + 1][lane], s_r[3 * warp + 2][lane]};
    const double m = q.st.m[i];
    if (q.precision == NB_FP64) {
        double4_32a *const dst[4] = {q.rec64.x, q.rec64.v, q.rec64.ab, q.rec64.kb};
        dst[warp][i] = make_double4_32a(r[0], r[1], r[2], warp == 0 ? m : 0.0);
    } else if (warp == 0) {
        float hi[3], lo[3], u[3];
        split_record(r, r, hi, lo, u);
        q.rec.ph[i] = make_float4(hi[0], hi[1], hi[2], to_float_int(m));
        q.rec.pl[i] = make_float4(lo[0], lo[1], lo[2], 0.0f);
    } else {
        float4 *const dst = warp == 1 ? q.rec.v : (warp == 2 ? q.rec.ab : q.rec.kb);
        dst[i] = make_float4(to_float_int(r[0]), to_float_int(r[1]), to_float_int(r[2]), 0.0f);
    }
}

// Copies of the FP64 state (checkpoints).
__global__ void k_copy_state(State dst, State src)
{
    const long long n3 = 3LL * src.n;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n3;
         e += (long long)gridDim.x * blockDim.x) {
        dst.x[e] = src.x[e];
        dst.v[e] = src.v[e];
        dst.a[e] = src.a[e];
        dst.k[e] = src.k[e];
    }
}

int grid_for(long long n, int nt)
{
    long long g = (n + nt - 1) / nt;
    return (int)(g < 1 ? 1 : (g > 4096 ? 4096 : g));
}

}  // namespace

int vjp_slots(int precision, int sms)
{
    int b = 0;
    cudaError_t e = precision == NB_FP64
                        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_force_vjp_f64<true>, kVNT, 0)
                        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, k_force_vjp_ds<2, true>, kVDsNT, 0);
    return e == cudaSuccess ? sms * (b > 0 ? b : 1) : sms;
}

int launch_force_vjp(const VjpArgs &va_in, int precision, bool softened, bool combine, int *slices,
                     cudaStream_t st)
{
    VjpArgs va = va_in;
    if (precision == NB_FP64) {
        va.plan = plan_ipar(va.n, va.n, kVNT, kVNT, va.slots, 0, va.part_cap);
        const int g = va.plan.items < va.slots ? va.plan.items : va.slots;
        if (softened) k_force_vjp_f64<true><<<g, kVNT, 0, st>>>(va);
        else k_force_vjp_f64<false><<<g, kVNT, 0, st>>>(va);
    } else {
        int R = 2;
        va.plan = plan_vjp_ds(va.n, va.slots, va.part_cap, R);
        const int g = va.plan.items;
        if (R == 1) {
            if (softened) k_force_vjp_ds<1, true><<<g, kVDsNT, 0, st>>>(va);
            else k_force_vjp_ds<1, false><<<g, kVDsNT, 0, st>>>(va);
        } else {
            if (softened) k_force_vjp_ds<2, true><<<g, kVDsNT, 0, st>>>(va);
            else k_force_vjp_ds<2, false><<<g, kVDsNT, 0, st>>>(va);
        }
    }
    const Plan P = va.plan;
    int launches = 1;
    // without the combine the caller adds the slices, in slice order
    if (slices) *slices = combine ? 1 : P.S;
    if (P.S > 1 && combine) {
        k_vjp_combine<<<grid_for(7LL * va.n, 256), 256, 0, st>>>(va, P.S);
        ++launches;
    }
    return launches;
}

void launch_shared_step(const SharedStep &q, cudaStream_t st)
{
    k_shared_step<<<cdiv(q.src.n, kShP), kShNT, 0, st>>>(q);
}

void launch_shared_done(const State &s, Ctrl *ctrl, int *act, long long steps, int level, cudaStream_t st)
{
    k_shared_done<<<grid_for(s.n, 256), 256, 0, st>>>(s, ctrl, act, steps, level);
    k_shared_ctrl<<<1, 1, 0, st>>>(ctrl, s.n, steps, level);
}

void launch_shared_times(const State &s, long long t, int level, cudaStream_t st)
{
    k_shared_times<<<grid_for(s.n, 256), 256, 0, st>>>(s, t, level);
}

void launch_adj_step(const AdjStep &q, cudaStream_t st)
{
    k_adj_step<<<cdiv(q.st.n, kShP), kShNT, 0, st>>>(q);
}

void launch_adj_pre(const State &s, double dt, const double *xb, const double *vb, double *ab,
                    double *kb, int precision, const VjpRecDS &rec, const VjpRec64 &rec64,
                    cudaStream_t st)
{
    k_adj_pre<<<grid_for(s.n, 128), 128, 0, st>>>(s, dt, xb, vb, ab, kb, precision, rec, rec64);
}

void launch_adj_post(int n, double dt, double *xb, double *vb, double *ab, double *kb, double *mb,
                     const double *xg, const double *vg, const double *mg, cudaStream_t st)
{
    k_adj_post<<<grid_for(n, 256), 256, 0, st>>>(n, dt, xb, vb, ab, kb, mb, xg, vg, mg);
}

void launch_adj_initial_rec(const State &s, const double *ab, const double *kb, int precision,
                            const VjpRecDS &rec, const VjpRec64 &rec64, cudaStream_t st)
{
    k_adj_initial_rec<<<grid_for(s.n, 256), 256, 0, st>>>(s, ab, kb, precision, rec, rec64);
}

void launch_add3(int n, double *dst, const double *src, double *dst2, const double *src2,
                 double *dstm, const double *srcm, cudaStream_t st)
{
    k_add3<<<grid_for(n, 256), 256, 0, st>>>(n, dst, src, dst2, src2, dstm, srcm);
}

void launch_set_ak(const State &s, const double *acc, const double *jerk, cudaStream_t st)
{
    k_set_ak<<<grid_for(s.n, 256), 256, 0, st>>>(s, acc, jerk);
}

void launch_copy_state(const State &dst, const State &src, cudaStream_t st)
{
    k_copy_state<<<grid_for(3LL * src.n, 256), 256, 0, st>>>(dst, src);
}

}  // namespace nbk
