// k_noalloc.cu -- force on a few particles with no device allocation at all.
//
// Some callers cannot allocate device memory when they need a force: a host
// application that hands this library a fixed slice of GPU memory and forbids
// later cudaMalloc calls, a real-time loop in which an allocation could block
// or fail, or a plug-in whose host owns the device allocator.  For them
// nb_force_few_noalloc evaluates the force on up to NB_NOALLOC_MAX_ACTIVE
// particles straight from the caller's FP64 arrays, with no context.  Its
// only working memory is the file-scope array below, which the runtime places
// on each GPU when the library's module is loaded there and keeps until the
// process exits.
//
// The sums are fixed as runs: the j range falls into slices (as many as give
// two per SM for four active particles a CTA), a slice into groups of 2048 j,
// and run t of a group is the plain FP32 sum of its pairs with j = t, t + 256,
// ... (at most eight).  Everything beyond a run is added in double-single or
// FP64, so which thread adds which run does not show in single precision.
//
// A CTA takes a range of groups and up to 64 active particles.  Each thread
// loads its eight j of a group straight from the FP64 arrays and splits them
// into double-single form once, in registers, then walks the active particles
// (in shared memory): eight pairs, and a warp reduce-scatter into the warp's
// double-single totals (k_few_partials).  Where the particles fill the lanes of a
// warp, they take the lanes and the runs the warps instead (k_few_lanes), without
// the reductions (27 of the 63 instructions a pair).  Both are bound by issue.
// The CTA adds its warps and writes one FP64 partial per value; a second kernel
// adds the ranges, a warp per value.  Every partial is written before it is
// read in the same call, so nothing in the scratch array needs clearing between
// calls.
//
// The first form held four active particles per CTA and split every j again
// for each four, on the FP64 pipe: 16 conversions a j at 2 lanes a clock per
// SM were nearly all of its time (64 active on 2^18 + 37 bodies: 148 us; 49 with
// the split once a CTA, 41 with the particles over the lanes).
#include <algorithm>
#include <climits>
#include <cmath>
#include <mutex>

#include "nb.h"
#include "nb_device.cuh"

namespace {

constexpr int kNT = 256;                    // threads per CTA
constexpr int kIC = 4;                      // active particles that the slice count is chosen for
constexpr int kComp = 7;                    // acc xyz, jerk xyz, pot
constexpr int kMaxSlices = 2048;            // j slices, and j ranges, at most
constexpr int kRun = 8;                     // FP32 pair terms per run
constexpr int kGroup = kNT * kRun;          // j per group of runs
constexpr long long kScratchDoubles = (long long)kMaxSlices * kComp * NB_NOALLOC_MAX_ACTIVE;
constexpr int kMaxDevices = 64;

// Partials of the j ranges: part[(b * 7 + c) * n_active + a].  7 MiB per GPU.
static __device__ __align__(256) double g_scratch[kScratchDoubles];

using nbk::dev::ds_add;
using nbk::dev::IDS;
using nbk::dev::make_ids;
using nbk::dev::pair_ds_packed;
using nbk::dev::rsqrt_sfu;
using nbk::dev::split_record;
using nbk::dev::to_float_int;
using nbk::dev::two_sum_acc;
using nbk::dev::warp_reduce_scatter;

struct DSPoint {
    float xh[3], xl[3], v[3], m;
};

__device__ __forceinline__ DSPoint load_point(const double *m, const double *x, const double *v,
                                              long long j)
{
    DSPoint p;
    const double xj[3] = {x[3 * j], x[3 * j + 1], x[3 * j + 2]}, vj[3] = {v[3 * j], v[3 * j + 1], v[3 * j + 2]};
    split_record(xj, vj, p.xh, p.xl, p.v);
    p.m = to_float_int(m[j]);
    return p;
}

// FP32 pair terms (Eq. 1 with the pair terms of the Appendix A kernel) on
// double-single positions; a pair to be skipped and, with eps = 0, any pair at
// r = 0 contribute nothing.  (Packing two j an instruction outside the running
// sums left 64 active on 2^18 + 37 bodies at 52.1 against 50.5 us: about half
// the instructions are the warp reductions', and the registers spill.)
__device__ __forceinline__ void pair(const DSPoint &J, const DSPoint &I, float eps2, bool skip,
                                     float acc[3], float jk[3], float &pot)
{
    float d[3], u[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        d[c] = (J.xh[c] - I.xh[c]) + (J.xl[c] - I.xl[c]);
        u[c] = J.v[c] - I.v[c];
    }
    const float r2 = fmaf(d[0], d[0], fmaf(d[1], d[1], fmaf(d[2], d[2], eps2)));
    const float rv = fmaf(d[0], u[0], fmaf(d[1], u[1], d[2] * u[2]));
    float rinv = rsqrt_sfu(r2);
    rinv = (skip || !(r2 > 0.0f)) ? 0.0f : rinv;
    const float rinv2 = rinv * rinv;
    const float mr = J.m * rinv;
    const float mr3 = mr * rinv2;
    const float b = -3.0f * rv * rinv2;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        acc[c] = fmaf(mr3, d[c], acc[c]);
        jk[c] = fmaf(mr3, fmaf(b, d[c], u[c]), jk[c]);
    }
    pot -= mr;
}

// CTA (b, ch): j groups [b G / B, (b + 1) G / B) of the G = S gps groups (gps a
// slice), active particles [ch IC, (ch + 1) IC).
__global__ void __launch_bounds__(kNT, 2) k_few_partials(long long n, const double *m, const double *x,
                                                         const double *v, float eps2, const int *act,
                                                         int na, long long jslice, int gps, long long G,
                                                         int B, int IC, int chunks, double *part)
{
    constexpr int NW = kNT / 32;
    constexpr int NV = NB_NOALLOC_MAX_ACTIVE * kComp;
    __shared__ DSPoint s_i[NB_NOALLOC_MAX_ACTIVE];
    __shared__ long long s_ii[NB_NOALLOC_MAX_ACTIVE];
    __shared__ float s_h[NW][NV], s_l[NW][NV];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int ch = blockIdx.x % chunks, b = blockIdx.x / chunks;
    const int cnt = min(IC, na - ch * IC);
    if (tid < cnt) {
        long long i = act[ch * IC + tid];
        i = i < 0 ? 0 : (i >= n ? n - 1 : i);
        s_ii[tid] = i;
        s_i[tid] = load_point(m, x, v, i);
    }
    for (int e = lane; e < cnt * kComp; e += 32) s_h[warp][e] = s_l[warp][e] = 0.0f;
    __syncthreads();
    const long long g1 = (b + 1) * G / B;
    for (long long g = b * G / B; g < g1; ++g) {
        const long long sl = g / gps;
        const long long j0 = sl * jslice + (g - sl * gps) * kGroup;
        const long long j1 = (sl + 1) * jslice < n ? (sl + 1) * jslice : n;
        if (j0 >= j1) continue;   // past the end of a short slice
        DSPoint jp[kRun];
#pragma unroll
        for (int u = 0; u < kRun; ++u) {
            const long long j = j0 + u * kNT + tid;
            jp[u] = load_point(m, x, v, j < j1 ? j : j1 - 1);
        }
        const int left = (int)(j1 - j0 < kGroup ? j1 - j0 : kGroup);   // j of this group
        for (int a = 0; a < cnt; ++a) {
            const DSPoint I = s_i[a];
            // this thread's j that is the particle itself, as a run position
            const long long own = s_ii[a] - j0 - tid;
            float a3[3] = {0.0f, 0.0f, 0.0f}, k3[3] = {0.0f, 0.0f, 0.0f}, pp = 0.0f;
            if (left < kGroup || (unsigned long long)(s_ii[a] - j0) < (unsigned long long)kGroup) {
#pragma unroll
                for (int u = 0; u < kRun; ++u)
                    pair(jp[u], I, eps2, u * kNT + tid >= left || own == u * kNT, a3, k3, pp);
            } else {
#pragma unroll
                for (int u = 0; u < kRun; ++u) pair(jp[u], I, eps2, false, a3, k3, pp);
            }
            float h[8] = {a3[0], a3[1], a3[2], k3[0], k3[1], k3[2], pp, 0.0f};
            float lo[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            warp_reduce_scatter<8>(h, lo, lane);
            const int e = lane >> 2;
            if ((lane & 3) == 0 && e < kComp)
                ds_add(s_h[warp][a * kComp + e], s_l[warp][a * kComp + e], h[0], lo[0]);
        }
    }
    __syncthreads();
    for (int t = tid; t < cnt * kComp; t += kNT) {
        float th = s_h[0][t], tl = s_l[0][t];
#pragma unroll
        for (int ww = 1; ww < NW; ++ww) ds_add(th, tl, s_h[ww][t], s_l[ww][t]);
        const int q = t / kComp, c = t % kComp;
        part[((long long)b * kComp + c) * na + ch * IC + q] = (double)th + (double)tl;
    }
}

// The same with the active particles over the lanes (R a lane) and
// the runs over the warps: a run's sum is added to its lane's totals by one TwoSum
// a value, where the form above needs a warp reduction of every run.  A CTA takes
// the items [b W / B, (b + 1) W / B) of W = 16 G: the runs t0 .. t0 + 15 of a group,
// 128 j, split once into shared memory (the next item's are on their way from
// memory meanwhile) and read by broadcast.
constexpr int kItemRuns = 16;               // runs of an item
constexpr int kItemJ = kItemRuns * kRun;    // its j
constexpr int kGroupItems = kNT / kItemRuns;

template <int R>
__global__ void __launch_bounds__(kNT, 2) k_few_lanes(long long n, const double *m, const double *x, const double *v,
                                                      float eps2, const int *act, int na, long long jslice, int gps,
                                                      long long G, double *part)
{
    constexpr int NW = kNT / 32, NV = 32 * R * kComp;
    __shared__ float4 s_j[2][3][kItemJ];
    __shared__ float s_h[NW][NV], s_l[NW][NV];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, b = blockIdx.x, B = gridDim.x;
    long long ii[R];
    IDS I[R];
    float hi[R][kComp], lo[R][kComp];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int a = 32 * r + lane;
        const long long i = act[a < na ? a : 0];
        ii[r] = i < 0 ? 0 : (i >= n ? n - 1 : i);
        const DSPoint p = load_point(m, x, v, ii[r]);
        I[r] = make_ids(make_float4(p.xh[0], p.xh[1], p.xh[2], p.m), make_float4(p.xl[0], p.xl[1], p.xl[2], 0.0f),
                        make_float4(p.v[0], p.v[1], p.v[2], 0.0f));
#pragma unroll
        for (int c = 0; c < kComp; ++c) hi[r][c] = lo[r][c] = 0.0f;
    }
    const long long w1 = (b + 1) * G * kGroupItems / B;
    double xj[3], vj[3], mj = 0.0;
    // this thread's j of item w (past the end: the last one, whose pairs are not formed)
    const auto fetch = [&](long long w) {
        const long long g = w / kGroupItems, sl = g / gps;
        const long long j1 = (sl + 1) * jslice < n ? (sl + 1) * jslice : n;
        long long j = sl * jslice + (g - sl * gps) * kGroup + (w % kGroupItems) * kItemRuns +
                      (tid / kItemRuns) * kNT + tid % kItemRuns;
        j = j < j1 ? j : j1 - 1;
#pragma unroll
        for (int c = 0; c < 3; ++c) xj[c] = x[3 * j + c], vj[c] = v[3 * j + c];
        mj = m[j];
    };
    long long w = b * G * kGroupItems / B;
    if (tid < kItemJ && w < w1) fetch(w);
    for (int buf = 0; w < w1; ++w, buf ^= 1) {
        if (tid < kItemJ) {
            float h[3], l[3], u[3];
            split_record(xj, vj, h, l, u);
            s_j[buf][0][tid] = make_float4(h[0], h[1], h[2], to_float_int(mj));
            s_j[buf][1][tid] = make_float4(l[0], l[1], l[2], 0.0f);
            s_j[buf][2][tid] = make_float4(u[0], u[1], u[2], 0.0f);
        }
        __syncthreads();
        if (tid < kItemJ && w + 1 < w1) fetch(w + 1);
        const long long g = w / kGroupItems, sl = g / gps;
        const long long j0 = sl * jslice + (g - sl * gps) * kGroup;
        const long long j1 = (sl + 1) * jslice < n ? (sl + 1) * jslice : n;
        const int left = (int)(j1 - j0 < kGroup ? j1 - j0 : kGroup);   // at most 0 past a short slice
        int own[R];   // the particle's position in the group
#pragma unroll
        for (int r = 0; r < R; ++r)
            own[r] = (unsigned long long)(ii[r] - j0) < (unsigned long long)kGroup ? (int)(ii[r] - j0) : -1;
#pragma unroll 1
        for (int q = 0; q < kItemRuns / NW; ++q) {
            const int tt = warp * (kItemRuns / NW) + q, t = (int)(w % kGroupItems) * kItemRuns + tt;
            float a3[R][3], k3[R][3], pp[R];
            bool mine = false;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                a3[r][0] = a3[r][1] = a3[r][2] = k3[r][0] = k3[r][1] = k3[r][2] = pp[r] = 0.0f;
                mine |= own[r] >= 0 && ((own[r] - t) & (kNT - 1)) == 0;
            }
            if (t + (kRun - 1) * kNT >= left || __any_sync(0xffffffffu, mine)) {
#pragma unroll 1
                for (int u = 0; u < kRun && t + u * kNT < left; ++u) {
                    const int e = u * kItemRuns + tt;
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        pair_ds_packed<false, true>(s_j[buf][0][e], s_j[buf][1][e], s_j[buf][2][e], I[r], eps2, a3[r],
                                                    k3[r], pp[r], t + u * kNT, own[r]);
                }
            } else {
#pragma unroll
                for (int u = 0; u < kRun; ++u) {
                    const int e = u * kItemRuns + tt;
                    const float4 p = s_j[buf][0][e], l = s_j[buf][1][e], d = s_j[buf][2][e];
#pragma unroll
                    for (int r = 0; r < R; ++r)
                        pair_ds_packed<false, false>(p, l, d, I[r], eps2, a3[r], k3[r], pp[r]);
                }
            }
#pragma unroll
            for (int r = 0; r < R; ++r)
#pragma unroll
                for (int c = 0; c < kComp; ++c)
                    two_sum_acc(hi[r][c], lo[r][c], c < 3 ? a3[r][c] : (c < 6 ? k3[r][c - 3] : pp[r]));
        }
    }
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
        for (int c = 0; c < kComp; ++c) {
            s_h[warp][(32 * r + lane) * kComp + c] = hi[r][c];
            s_l[warp][(32 * r + lane) * kComp + c] = lo[r][c];
        }
    __syncthreads();
    for (int t = tid; t < na * kComp; t += kNT) {
        float th = s_h[0][t], tl = s_l[0][t];
#pragma unroll
        for (int ww = 1; ww < NW; ++ww) ds_add(th, tl, s_h[ww][t], s_l[ww][t]);
        part[((long long)b * kComp + t % kComp) * na + t / kComp] = (double)th + (double)tl;
    }
}

// One warp per value: lanes over the ranges in a fixed stride, then a fixed
// tree (one thread per value, adding the ranges in turn, waited for its loads
// four at a time: ~15 us for one active particle on 2^18 bodies).
__global__ void k_few_combine(int na, int B, const double *part, double *acc, double *jerk,
                              double *pot)
{
    const int lane = threadIdx.x & 31;
    const int e = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (e >= na * kComp) return;
    const int c = e / na, a = e % na;
    double s = 0.0;
#pragma unroll 4
    for (int q = lane; q < B; q += 32) s += part[((long long)q * kComp + c) * na + a];
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) s += __shfl_xor_sync(0xffffffffu, s, off);
    if (lane != 0) return;
    if (c < 3) {
        if (acc) acc[3 * a + c] = s;
    } else if (c < 6) {
        if (jerk) jerk[3 * a + (c - 3)] = s;
    } else if (pot) {
        pot[a] = s;
    }
}

// Per-device set-up: the device address of g_scratch (host code may not use
// the symbol itself, which on the host is only a stand-in) and the SM count.
struct DeviceSetup {
    double *scratch = nullptr;
    int sms = 0;
};
DeviceSetup g_setup[kMaxDevices];
std::mutex g_setup_mutex;

int setup_current_device(DeviceSetup *out)
{
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return NB_ECUDA;
    std::lock_guard<std::mutex> lock(g_setup_mutex);
    DeviceSetup &s = g_setup[dev];
    if (!s.scratch) {
        void *p = nullptr;
        if (cudaGetSymbolAddress(&p, g_scratch) != cudaSuccess || !p) {
            cudaGetLastError();
            return NB_ECUDA;
        }
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
            cudaGetLastError();
            return NB_ECUDA;
        }
        s.sms = sms > 0 ? sms : 1;
        s.scratch = (double *)p;
    }
    *out = s;
    return NB_OK;
}

}  // namespace

extern "C" int nb_force_few_noalloc(int64_t n, const double *d_m, const double *d_x,
                                    const double *d_v, double eps, const int32_t *d_active_idx,
                                    int32_t n_active, double *d_acc, double *d_jerk, double *d_pot,
                                    void *stream)
{
    if (n < 1 || n > INT_MAX) return NB_EINVAL;
    if (n_active < 0 || n_active > NB_NOALLOC_MAX_ACTIVE) return NB_EINVAL;
    if (!std::isfinite(eps) || eps < 0.0) return NB_EINVAL;
    if (n_active == 0) return NB_OK;
    if (!d_m || !d_x || !d_v || !d_active_idx) return NB_EINVAL;
    // An error left pending by earlier work is not this call's: report it
    // without launching and without clearing it.
    if (cudaPeekAtLastError() != cudaSuccess) return NB_ECUDA;
    DeviceSetup s;
    const int rc = setup_current_device(&s);
    if (rc != NB_OK) return rc;

    // Slices: about two CTAs per SM in total, at least eight j per thread,
    // at most kMaxSlices (so the partials fit the scratch array).
    const int chunks = (n_active + kIC - 1) / kIC;
    long long S = (2LL * s.sms + chunks - 1) / chunks;
    const long long smax = (n + 8LL * kNT - 1) / (8LL * kNT);
    if (S > smax) S = smax;
    if (S > kMaxSlices) S = kMaxSlices;
    if (S < 1) S = 1;
    const long long jslice = ((n + S - 1) / S + kNT - 1) / kNT * kNT;
    S = (n + jslice - 1) / jslice;
    // Work: G groups of runs by the active particles, two CTAs resident an SM.
    // With fewer groups than CTAs the particles are divided too, no further than
    // one round of CTAs (each splits its j again: 64 active on 2^18 + 37 bodies
    // take 49 us so, 55 and 66 us with two and four times the CTAs); otherwise
    // a CTA takes several groups.
    const int gps = (int)((jslice + kGroup - 1) / kGroup);
    const long long G = S * gps, slots = 2LL * s.sms;
    const long long rounds = (G + slots - 1) / slots;
    int B = (int)((G + rounds - 1) / rounds);
    int parts = (int)(slots / B < n_active ? slots / B : n_active);
    if (parts < 1) parts = 1;
    const int IC = (n_active + parts - 1) / parts;
    const int ichunks = (n_active + IC - 1) / IC;

    cudaStream_t st = (cudaStream_t)stream;
    // Particles over the lanes where nearly all lanes have one.  This form / the one
    // with the runs over the lanes, us, on 2^18 + 37 bodies: 24 active 31.2 / 27.1,
    // 32 31.2 / 31.2, 48 41.5 / 39.4, 64 41.5 / 48.7; on 2^20: 24 82.5 / 70.1,
    // 32 78.4 / 86.5, 48 123.5 / 119.3, 64 119.5 / 150.0.
    const int R = (n_active + 31) / 32;
    const bool lanes = 16 * n_active >= 15 * 32 * R;
    if (lanes) {
        const long long W = G * kGroupItems;
        B = (int)std::min<long long>(W, std::min<long long>(slots, kMaxSlices));
        const auto kernel = R == 1 ? k_few_lanes<1> : k_few_lanes<2>;
        kernel<<<B, kNT, 0, st>>>(n, d_m, d_x, d_v, (float)(eps * eps), d_active_idx, n_active, jslice, gps, G,
                                  s.scratch);
    } else {
        k_few_partials<<<B * ichunks, kNT, 0, st>>>(n, d_m, d_x, d_v, (float)(eps * eps), d_active_idx,
                                                    n_active, jslice, gps, G, B, IC, ichunks, s.scratch);
    }
    if (cudaGetLastError() != cudaSuccess) return NB_ECUDA;
    k_few_combine<<<(n_active * kComp * 32 + 255) / 256, 256, 0, st>>>(n_active, B, s.scratch, d_acc,
                                                                       d_jerk, d_pot);
    return cudaGetLastError() == cudaSuccess ? NB_OK : NB_ECUDA;
}
