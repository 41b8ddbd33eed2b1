// k_ensemble.cu -- many independent clusters advanced together: every
// ensemble block step advances every unfinished cluster by its own next block
// step (Section 2 step loop: select the block, predict, force, correct) in
// three launches, replayed from CUDA graphs:
//   k_ens_sched, a CTA per cluster, largest first: block time t_next = min over
//      the cluster of t_i + dt_i, the block compacted in ascending order, a
//      force item per chunk of active particles queued by size class, and up to
//      512 particles predicted to t_next (predict_j32: FP32 increments on a
//      single-precision mirror, into double-single j records);
//   k_ens_predict: the prediction of larger clusters, a CTA per 512 particles;
//   k_ens_force: the force items, the largest clusters' first, drawn by CTAs
//      that fill the GPU: g lanes share one or two active particles and split
//      the j (FP32 pair arithmetic on double-single positions, TwoSum-promoted
//      sums), then four lanes correct a particle (FP64 corrector and Aarseth
//      step).  The force reads only the j records, so correcting while other
//      items still sum is safe.
// Nothing waits inside a launch, and every particle's sums are formed in an order
// that only (threads, gmax) fix, so results do not depend on which CTA takes an item.
//
// 256 clusters of 32..4096, a mean of 2e7 pairs a step: 70 us a step (start-up
// of a graph included: 73 with one step a graph), of which k_ens_sched 6.3,
// k_ens_predict 4, k_ens_force 37-45, the gaps between launches 2.3 each.  One
// cooperative launch with queues between the phases took 125 us: its items
// computed all of the CTA's lane groups, active or not, and their CTAs waited for
// the correction; with lone particles' warps leaving early and the j of a large
// cluster shared by ways 80, as three launches 76.  All particles active, the force
// runs at 7e11 pairs/s, bound by instruction issue (44 a pair and lane) and by shared
// memory (6.4 wavefronts; one particle a lane: 5.5e11, 52 and 12.9).
#include <algorithm>
#include <climits>
#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include <nvtx3/nvToolsExt.h>

#include "nb_device.cuh"
#include "nb_int64.cuh"

namespace nbk {
namespace {

using namespace dev;

constexpr int kEnsMaxN = 4096;       // largest cluster
constexpr int kEnsPredChunk = 512;   // larger clusters are predicted in chunks by several CTAs
constexpr int kEnsClasses = 4;       // force items by cluster size, the longest first

__host__ __device__ inline int ens_class(int n) { return n > 2048 ? 0 : (n > 1024 ? 1 : (n > 512 ? 2 : 3)); }

constexpr int kEnsANT = 256;         // threads of a scheduling CTA
constexpr int kEnsPNT = 128;         // ... of a prediction CTA
constexpr int kEnsFNT = 128;         // ... of a force CTA
constexpr int kEnsR = 2;             // active particles of a lane group, large blocks
constexpr int kEnsMaxWays = 2;       // sum blocks that a force CTA works on at once (see ens_sums)
constexpr int kEnsChain = 2048;      // a cluster above this many j has its force items cut for two ways
constexpr int kEnsStageJ = 256;      // j of a stage
constexpr int kEnsStages = 2;
constexpr int kEnsGraphSteps = 8;    // steps of the longer graph

struct EnsArgs {
    int C;                    // clusters
    const long long *off;     // [C + 1] particle offsets
    const int *order;         // clusters in decreasing size
    State s;                  // all particles, SoA over the total count
    float eps2;
    double eta, eta_init;
    int level_min;
    long long t_end;
    int g;                    // lanes per active particle
    int sb;                   // j of a sum block
    int *work;                // counters: force items claimed, force CTAs done, and the queue
                              // lengths [kEnsClasses]; all 0 between launches
    const int2 *pitem;        // prediction items: cluster, chunk
    int2 *queue;              // force items: cluster, chunk; [P] in size classes
    int qbase[kEnsClasses];   // first slot of each class
    float4 *jph, *jpl, *jv;   // [P] predicted double-single records
    Mirror mir;               // [P] single-precision mirror of the FP64 state for the j predictor
    int *act;                 // [P] active particles of each cluster (local indices)
    int *na;                  // [C] block sizes
    long long *tnext;         // [C] block times
    int *done;                // [C]
    long long *steps;         // [C]
    long long *inter;         // [C] sum of n_active (n - 1)
    int *err;
    double *out_acc, *out_jerk, *out_pot;  // force-only mode: [P][3], [P][3], [P]
};

// Ways and particles of a full force item of a cluster.  Two ways above 2048 j:
// 512 launches of 256 clusters of 32..4096 take 37.9 ms with the line there, 38.6
// at 1024 or 512, 42.6 without it, 41.9 with four ways above 1024 (the items
// read their j from the L2 cache, so smaller ones read more).
__device__ __forceinline__ int ens_ways(int n) { return n > kEnsChain ? kEnsMaxWays : 1; }
__device__ __forceinline__ int ens_chunk(int n, int na, int g)
{
    const int one = kEnsFNT / g / ens_ways(n);
    return na > one ? kEnsR * one : one;
}

template <typename T, typename Op>
__device__ __forceinline__ T cta_reduce(T v, Op op, T *smem)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int o = 16; o >= 1; o >>= 1) v = op(v, __shfl_xor_sync(0xffffffffu, v, o));
    __syncthreads();
    if (lane == 0) smem[warp] = v;
    __syncthreads();
    T r = smem[0];
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) r = op(r, smem[w]);
    __syncthreads();
    return r;
}

struct MinLL {
    __device__ long long operator()(long long a, long long b) const { return a < b ? a : b; }
};

enum EnsMode { kEnsStep = 0, kEnsForce = 1, kEnsInit = 2 };

// j record of particle gi at block time tn from the single-precision mirror
// (predict_j32: FP32 Taylor increments, double-single position add).  The FP64
// state itself is predicted in FP64 by the corrector.
__device__ __forceinline__ void ens_predict_j32(const EnsArgs &ea, long long gi, long long tn)
{
    float4 ph, pl, pv;
    predict_j32(ea.mir, gi, tn - ea.s.t[gi], ph, pl, pv);
    ea.jph[gi] = ph;
    ea.jpl[gi] = pl;
    ea.jv[gi] = pv;
}

__device__ __forceinline__ void ens_write_mirror(const EnsArgs &ea, long long gi)
{
    write_mirror(ea.s, ea.mir, gi, ea.s.n);
}

__global__ void k_ens_mirror(EnsArgs ea)
{
    for (long long gi = blockIdx.x * (long long)blockDim.x + threadIdx.x; gi < ea.s.n;
         gi += (long long)gridDim.x * blockDim.x)
        ens_write_mirror(ea, gi);
}

// The j record of the stored state itself (start-up and force-only passes: dt = 0).
__device__ __forceinline__ void ens_record(const EnsArgs &ea, long long gi)
{
    const State &S = ea.s;
    const long long P = S.n;
    float hi[3], lo[3];
#pragma unroll
    for (int cc = 0; cc < 3; ++cc) split_ds(S.x[cc * P + gi], hi[cc], lo[cc]);
    ea.jph[gi] = make_float4(hi[0], hi[1], hi[2], __double2float_rn(S.m[gi]));
    ea.jpl[gi] = make_float4(lo[0], lo[1], lo[2], 0.0f);
    ea.jv[gi] = make_float4(__double2float_rn(S.v[gi]), __double2float_rn(S.v[P + gi]),
                            __double2float_rn(S.v[2 * P + gi]), 0.0f);
}

struct AShared {
    long long red[16];
    unsigned bal[kEnsMaxN / 32];
    int off[kEnsMaxN / 32];
    int base;
};

// Schedules the cluster of rank blockIdx.x: block time, block, force items; a small
// cluster is predicted as well.  The
// next times are read once, into shared memory, and the block is compacted with
// one ballot word per 32 particles and one scan of the words.
template <int MODE>
__global__ void __launch_bounds__(kEnsANT) k_ens_sched(EnsArgs ea)
{
    constexpr int NT = kEnsANT;
    __shared__ AShared A;
    __shared__ long long s_next[kEnsMaxN];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const State &S = ea.s;
    const int c = ea.order[blockIdx.x];
    const long long o = ea.off[c];
    const int n = (int)(ea.off[c + 1] - o);
    if (MODE == kEnsStep && ea.done[c]) return;
    long long tn = 0;
    if (MODE == kEnsStep) {
        long long mn = LLONG_MAX;
#pragma unroll 4
        for (int i = tid; i < n; i += NT) {
            const long long nx = S.t[o + i] + (1LL << (kTickBits - S.lev[o + i]));
            s_next[i] = nx;
            mn = min(mn, nx);
        }
        tn = cta_reduce(mn, MinLL(), A.red);
        if (tn > ea.t_end) {
            if (tid == 0) ea.done[c] = 1;
            return;
        }
    }
    const int words = (n + 31) >> 5;
    for (int w = warp; w < words; w += NT / 32) {
        const int i = 32 * w + lane;
        const unsigned bal = __ballot_sync(0xffffffffu, i < n && (MODE != kEnsStep || s_next[i] == tn));
        if (lane == 0) A.bal[w] = bal;
    }
    const bool split = n > kEnsPredChunk;  // prediction left to items of its own
    if (!split)
        for (int i = tid; i < n; i += NT) {
            if (MODE == kEnsStep) ens_predict_j32(ea, o + i, tn);
            else ens_record(ea, o + i);
        }
    __syncthreads();
    if (warp == 0) {
        constexpr int kPer = kEnsMaxN / 32 / 32;
        int cw[kPer], sum = 0;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            const int w = kPer * lane + u;
            cw[u] = w < words ? __popc(A.bal[w]) : 0;
            sum += cw[u];
        }
        int inc = sum;
#pragma unroll
        for (int d = 1; d < 32; d <<= 1) {
            const int up = __shfl_up_sync(0xffffffffu, inc, d);
            inc += lane >= d ? up : 0;
        }
        int at = inc - sum;
#pragma unroll
        for (int u = 0; u < kPer; ++u) {
            A.off[kPer * lane + u] = at;
            at += cw[u];
        }
        const int na = __shfl_sync(0xffffffffu, inc, 31);
        if (lane == 0) {
            ea.na[c] = na;
            ea.tnext[c] = tn;
            if (MODE == kEnsStep) {
                ea.steps[c] += 1;
                ea.inter[c] += (long long)na * (n - 1);
            }
        }
        const int chunk = ens_chunk(n, na, ea.g), cls = ens_class(n), nforce = (na + chunk - 1) / chunk;
        int base = lane == 0 ? atomicAdd(&ea.work[2 + cls], nforce) : 0;
        base = ea.qbase[cls] + __shfl_sync(0xffffffffu, base, 0);
        for (int k = lane; k < nforce; k += 32) ea.queue[base + k] = make_int2(c, k);
    }
    __syncthreads();
    for (int w = warp; w < words; w += NT / 32) {
        const unsigned bal = A.bal[w];
        if (bal >> lane & 1) ea.act[o + A.off[w] + __popc(bal & ((1u << lane) - 1u))] = 32 * w + lane;
    }
}

// Predicts one chunk of 512 particles of a larger cluster to its block time.
template <int MODE>
__global__ void __launch_bounds__(kEnsPNT) k_ens_predict(EnsArgs ea)
{
    const int2 it = ea.pitem[blockIdx.x];
    if (MODE == kEnsStep && ea.done[it.x]) return;
    const long long o = ea.off[it.x];
    const int n = (int)(ea.off[it.x + 1] - o);
    const long long tn = ea.tnext[it.x];
    const int i1 = min(n, (it.y + 1) * kEnsPredChunk);
    for (int i = it.y * kEnsPredChunk + threadIdx.x; i < i1; i += kEnsPNT) {
        if (MODE == kEnsStep) ens_predict_j32(ea, o + i, tn);
        else ens_record(ea, o + i);
    }
}

__device__ __forceinline__ void copy16(float4 *dst, const float4 *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(dst)), "l"(src)
                 : "memory");
}

struct FShared {
    union {
        float4 j[kEnsStages][3][kEnsStageJ];
        float res[kEnsR * kEnsFNT][14];
    };
    float part[kEnsR][7][kEnsFNT];
    int it;
};

// Sums of the particles act[0 .. cnt) of a cluster (R to a lane group) into sh.res.
//
// A particle's sums are fixed by (g, sb): lane q of its g lanes adds the j
// = q, q + g, ... of a sum block of sb j in FP32, and the blocks are promoted in
// order.  So the blocks can be shared out: the CTA's lanes make up several ways,
// each takes every ways-th block, and the first way's lanes promote all of them.
// The j come in stages of one tile a way, kEnsStages - 1 stages ahead.
template <int R, bool SOFT>
__device__ __forceinline__ void ens_sums(const EnsArgs &ea, long long o, int n, const int *act, int cnt, FShared &sh)
{
    constexpr int NT = kEnsFNT;
    const int tid = threadIdx.x;
    const int g = ea.g, sb = ea.sb;
    int per = g;   // lanes of a way
    while (R * per < cnt * g) per <<= 1;
    const int ways = min(min(kEnsMaxWays, NT / per), n <= sb ? 1 : 2);
    const int T = min(sb, kEnsStageJ / ways);   // j of a tile, a divisor of sb
    const int lgT = 31 - __clz(T);
    const float4 *jph = ea.jph + o, *jpl = ea.jpl + o, *jv = ea.jv + o;
    int fb = 0, fr = 0, fs = 0;   // next fetch: first block, tile within it, stage
    auto fetch = [&]() {
        for (int t = tid; t < ways * T; t += NT) {
            const int j = fb + (t >> lgT) * sb + fr + (t & (T - 1));
            if (j < n) {
                copy16(&sh.j[fs][0][t], jph + j);
                copy16(&sh.j[fs][1][t], jpl + j);
                copy16(&sh.j[fs][2][t], jv + j);
            }
        }
        asm volatile("cp.async.commit_group;" ::: "memory");
        fs = fs == kEnsStages - 1 ? 0 : fs + 1;
        fr += T;
        if (fr == sb) {
            fr = 0;
            fb += ways * sb;
        }
    };
#pragma unroll
    for (int q = 1; q < kEnsStages; ++q) fetch();
    const int way = tid / per, grp = tid % per / g, lig = tid % g, slots = per / g;
    const bool work = way < ways && grp < cnt, valid = work && way == 0;
    const bool warp_work = __any_sync(0xffffffffu, work), warp_valid = __any_sync(0xffffffffu, valid);
    int i[R];
    IDS I[R];
    float hi[R][7], lo[R][7];
#pragma unroll
    for (int r = 0; r < R; ++r) {
        const int a = grp + r * slots;
        i[r] = act[a < cnt ? a : 0];
        I[r] = make_ids(jph[i[r]], jpl[i[r]], jv[i[r]]);
#pragma unroll
        for (int cc = 0; cc < 7; ++cc) hi[r][cc] = lo[r][cc] = 0.0f;
    }
    int buf = 0;
    for (int jb = 0; jb < n; jb += ways * sb) {
        float ta[R][3], tk[R][3], tp[R];
#pragma unroll
        for (int r = 0; r < R; ++r)
            ta[r][0] = ta[r][1] = ta[r][2] = tk[r][0] = tk[r][1] = tk[r][2] = tp[r] = 0.0f;
        for (int q = 0; q < sb && jb + q < n; q += T) {
            asm volatile("cp.async.wait_group %0;" ::"n"(kEnsStages - 2) : "memory");
            __syncthreads();
            fetch();
            const int jt = jb + way * sb + q, jn = work ? min(n - jt, T) : 0;
            if (warp_work) {
                const float4 *ph = sh.j[buf][0] + way * T, *pl = sh.j[buf][1] + way * T, *pv = sh.j[buf][2] + way * T;
                bool mine = false;
#pragma unroll
                for (int r = 0; r < R; ++r) mine |= (unsigned)(i[r] - jt) < (unsigned)T;
                if (__any_sync(0xffffffffu, mine)) {
#pragma unroll 1
                    for (int jj = lig; jj < jn; jj += g)
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            pair_ds_packed<SOFT, true>(ph[jj], pl[jj], pv[jj], I[r], ea.eps2, ta[r], tk[r], tp[r],
                                                       jt + jj, i[r]);
                } else {
#pragma unroll (R == 1 ? 4 : 2)
                    for (int jj = lig; jj < jn; jj += g) {
                        const float4 h = ph[jj], l = pl[jj], v = pv[jj];
#pragma unroll
                        for (int r = 0; r < R; ++r)
                            pair_ds_packed<SOFT, false>(h, l, v, I[r], ea.eps2, ta[r], tk[r], tp[r]);
                    }
                }
            }
            buf = buf == kEnsStages - 1 ? 0 : buf + 1;
        }
        if (ways > 1) {
            if (work && way > 0)
#pragma unroll
                for (int r = 0; r < R; ++r)
#pragma unroll
                    for (int cc = 0; cc < 7; ++cc)
                        sh.part[r][cc][tid] = cc < 3 ? ta[r][cc] : (cc < 6 ? tk[r][cc - 3] : tp[r]);
            __syncthreads();
        }
        if (valid)
#pragma unroll
            for (int r = 0; r < R; ++r) {
#pragma unroll
                for (int cc = 0; cc < 7; ++cc)
                    two_sum_acc(hi[r][cc], lo[r][cc], cc < 3 ? ta[r][cc] : (cc < 6 ? tk[r][cc - 3] : tp[r]));
                for (int w = 1; w < ways && jb + w * sb < n; ++w)
#pragma unroll
                    for (int cc = 0; cc < 7; ++cc)
                        two_sum_acc(hi[r][cc], lo[r][cc], sh.part[r][cc][w * per + tid]);
            }
    }
    __syncthreads();   // the j tiles are done with: their space takes the sums
    if (warp_valid) {
#pragma unroll
        for (int r = 0; r < R; ++r) {
            for (int d = 1; d < g; d <<= 1) {
#pragma unroll
                for (int cc = 0; cc < 7; ++cc) {
                    const float h2 = __shfl_xor_sync(0xffffffffu, hi[r][cc], d);
                    const float l2 = __shfl_xor_sync(0xffffffffu, lo[r][cc], d);
                    ds_add(hi[r][cc], lo[r][cc], h2, l2);
                }
            }
            if (valid && lig == 0 && grp + r * slots < cnt)
#pragma unroll
                for (int cc = 0; cc < 7; ++cc) {
                    sh.res[grp + r * slots][cc] = hi[r][cc];
                    sh.res[grp + r * slots][7 + cc] = lo[r][cc];
                }
        }
    }
    __syncthreads();
}

// Force item (c, k): force on one chunk of the cluster's block, then the
// correction (or the start-up levels, or plain output).
template <int MODE, bool SOFT>
__device__ __forceinline__ void ens_b_item(const EnsArgs &ea, int c, int k, FShared &sh)
{
    constexpr int NT = kEnsFNT;
    const int tid = threadIdx.x;
    const State &S = ea.s;
    const long long P = S.n;
    const long long o = ea.off[c];
    const int n = (int)(ea.off[c + 1] - o), na = ea.na[c];
    const int chunk = ens_chunk(n, na, ea.g), s0 = k * chunk, cnt = min(chunk, na - s0);
    if (cnt > kEnsFNT / ea.g / ens_ways(n)) ens_sums<kEnsR, SOFT>(ea, o, n, ea.act + o + s0, cnt, sh);
    else ens_sums<1, SOFT>(ea, o, n, ea.act + o + s0, cnt, sh);
    if constexpr (MODE == kEnsStep) {
        // four lanes correct a particle, one axis each; whole warps of particles
        const int q = tid & 3, ax = q < 3 ? q : 2;
        const long long tn = ea.tnext[c];
        for (int u0 = 0; u0 + (tid >> 5) * 8 < cnt; u0 += NT / 4) {
            const int u = u0 + (tid >> 2), uu = min(u, cnt - 1);
            const long long gi = o + ea.act[o + s0 + uu];
            const bool ok = correct_particle_quad(S, gi, P, tn, (double)sh.res[uu][ax] + (double)sh.res[uu][7 + ax],
                                                  (double)sh.res[uu][3 + ax] + (double)sh.res[uu][10 + ax], ea.eta,
                                                  ea.level_min, 0, u < cnt);
            __syncwarp();
            if (u < cnt && q == 0) {
                if (!ok) atomicCAS(ea.err, 0, NB_ESTEP);
                ens_write_mirror(ea, gi);
            }
        }
    } else for (int u = tid; u < cnt; u += NT) {
        const long long gi = o + ea.act[o + s0 + u];
        double res[7];
#pragma unroll
        for (int cc = 0; cc < 7; ++cc) res[cc] = (double)sh.res[u][cc] + (double)sh.res[u][7 + cc];
        if constexpr (MODE == kEnsForce) {
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) {
                ea.out_acc[3 * gi + cc] = res[cc];
                ea.out_jerk[3 * gi + cc] = res[3 + cc];
            }
            ea.out_pot[gi] = res[6];
        } else {
#pragma unroll
            for (int cc = 0; cc < 3; ++cc) {
                S.a[cc * P + gi] = res[cc];
                S.k[cc * P + gi] = res[3 + cc];
            }
            S.t[gi] = 0;
            int lv;
            if (!level_of(initial_dt(res, res + 3, ea.eta_init), ea.level_min, lv)) {
                atomicCAS(ea.err, 0, NB_ESTEP);
                lv = kTickBits;
            }
            S.lev[gi] = lv;
        }
    }
}

// The force items, the longest clusters' first.
template <int MODE, bool SOFT>
__global__ void __launch_bounds__(kEnsFNT, 4) k_ens_force(EnsArgs ea)
{
    __shared__ FShared s;
    int len[kEnsClasses];
#pragma unroll
    for (int cls = 0; cls < kEnsClasses; ++cls) len[cls] = ea.work[2 + cls];
    int it = blockIdx.x;
    for (;;) {
        int at = it, slot = -1;
#pragma unroll
        for (int cls = 0; cls < kEnsClasses; ++cls) {
            if (slot < 0 && at < len[cls]) slot = ea.qbase[cls] + at;
            at -= len[cls];
        }
        if (slot < 0) break;
        if (threadIdx.x == 0) s.it = (int)gridDim.x + atomicAdd(&ea.work[0], 1);
        const int2 f = ea.queue[slot];
        ens_b_item<MODE, SOFT>(ea, f.x, f.y, s);
        __syncthreads();
        it = s.it;
        __syncthreads();
    }
    // the last CTA leaves the counters at 0
    __syncthreads();
    if (threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&ea.work[1], 1) == (int)gridDim.x - 1) {
            __threadfence();
            for (int q = 0; q < 2 + kEnsClasses; ++q) ea.work[q] = 0;
        }
    }
}

// Energy of every cluster at its particles' own times (exact when the cluster
// is synchronised): kinetic from FP64 velocities, potential as the FP64 pair
// sum -sum_{i<j} m_i m_j / sqrt(r^2 + eps^2), in a fixed order.
//
// The pair sum is cut into tiles of 128 x 128 pairs (ti <= tj) of every cluster,
// one CTA each, for all SMs to share.  A pair's m_j / r is formed on the integer
// pipes (nb_int64.cuh) with one FP64 addition; a tile with a value out of that
// range takes 12 FP64 operations a pair, 1/sqrt being five on an FP32 seed.
// 256 clusters of 32..4096 (2.7e8 pairs), with the copies: 1.3 ms; 6.1 with every
// tile in FP64; 96 with one CTA per cluster, a square root and a division.

constexpr int kEnTile = 128;

__host__ __device__ inline long long en_items(int n)
{
    const long long t = (n + kEnTile - 1) / kEnTile;
    return t * (t + 1) / 2;
}

// 1/sqrt(x): the SFU's FP32 value y0 (relative error about 2^-22), then
// y0 + y0 e (1/2 + 3/8 e) with e = 1 - x y0^2, the series of (1 - e)^(-1/2)
// to second order (the next term is below 2^-66).  The FP64 <-> FP32 steps are
// bit moves: conversions run on the FP64 pipe.
__device__ __forceinline__ double rsqrt_pair(double x)
{
    if (!exponent_in<-70, 190>(x)) return rsqrt(x);
    const unsigned xh = (unsigned)__double2hiint(x), xl = (unsigned)__double2loint(x);
    const float y = rsqrt_sfu(__uint_as_float((xh - (896u << 20)) << 3 | xl >> 29));   // truncated
    const unsigned yb = __float_as_uint(y);
    const double y0 = __hiloint2double((int)((yb >> 3) + (896u << 20)), (int)(yb << 29));
    const double e = fma(-(x * y0), y0, 1.0);
    return fma(fma(e, 0.375, 0.5), y0 * e, y0);
}

// Potential of pair tile blockIdx.x: item[] holds each cluster's first tile.
__global__ void __launch_bounds__(kEnTile) k_ens_pairs(EnsArgs ea, const int *item, double eps2, double *part)
{
    __shared__ union JTile {
        double4_32a f;
        struct {
            long long m[4];
            unsigned e;
        } i;
        __device__ JTile() {}
    } s_j[kEnTile];
    __shared__ double s_red[kEnTile / 32];
    const State &S = ea.s;
    const long long P = S.n;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    int c = 0;   // the last cluster whose first tile is not past this one
    for (int hi = ea.C - 1; c < hi;) {
        const int mid = (c + hi + 1) / 2;
        if (item[mid] <= (int)blockIdx.x) c = mid;
        else hi = mid - 1;
    }
    const int k = blockIdx.x - item[c];
    int tj = (int)((sqrtf(8.0f * (float)k + 1.0f) - 1.0f) * 0.5f);
    while ((tj + 1) * (tj + 2) / 2 <= k) ++tj;
    while (tj * (tj + 1) / 2 > k) --tj;
    const int ti = k - tj * (tj + 1) / 2;
    const long long o = ea.off[c];
    const int n = (int)(ea.off[c + 1] - o);
    const int i0 = ti * kEnTile + warp * 32, i = i0 + lane, j0 = tj * kEnTile, jc = min(kEnTile, n - j0);
    double4_32a pj = make_double4_32a(0., 0., 0., 0.), pi = pj;
    if (tid < jc) {
        const long long gj = o + j0 + tid;
        pj = make_double4_32a(S.x[gj], S.x[P + gj], S.x[2 * P + gj], S.m[gj]);
    }
    if (i0 < n) {
        const long long gi = o + min(i, n - 1);
        pi = make_double4_32a(S.x[gi], S.x[P + gi], S.x[2 * P + gi], S.m[gi]);
    }
    const auto in_range = [](const double4_32a &p) {
        return i64::in_range(p.x) && i64::in_range(p.y) && i64::in_range(p.z) && i64::in_range(p.w);
    };
    double row = 0.0;
    // on the diagonal a warp starts past its own first particle
    const int q0 = ti == tj ? warp * 32 + 1 : 0;
    if (__syncthreads_and(i64::eps2_in_range(eps2) && in_range(pi) && in_range(pj))) {
        const i64::Fix x = i64::to_fix(pj.x), y = i64::to_fix(pj.y), z = i64::to_fix(pj.z);
        const i64::Num m = i64::to_num(pj.w);
        s_j[tid].i.m[0] = x.m;
        s_j[tid].i.m[1] = y.m;
        s_j[tid].i.m[2] = z.m;
        s_j[tid].i.m[3] = (long long)m.m;
        s_j[tid].i.e = (unsigned)(x.e & 255) | (unsigned)(y.e & 255) << 8 | (unsigned)(z.e & 255) << 16 |
                       (unsigned)m.e << 24;
        __syncthreads();
        const i64::Eps eps = i64::make_eps(eps2);
        const i64::Fix I[3] = {i64::to_fix(pi.x), i64::to_fix(pi.y), i64::to_fix(pi.z)};
        if (i0 < n)
#pragma unroll 1
            for (int q = q0; q < jc; ++q) {
                const unsigned e = s_j[q].i.e;
                i64::Num D[3], mj;
#pragma unroll
                for (int cc = 0; cc < 3; ++cc) {
                    i64::Fix X;
                    X.m = s_j[q].i.m[cc];
                    X.e = i64::signed_byte(e, cc);
                    double d;
                    D[cc] = i64::diff(X, I[cc], d);
                }
                mj.m = (unsigned long long)s_j[q].i.m[3];
                mj.e = i64::signed_byte(e, 3);
                mj.neg = false;
                const double v = i64::pair_potential(D, mj, eps);
                row += j0 + q > i ? v : 0.0;
            }
    } else {
        s_j[tid].f = pj;
        __syncthreads();
        if (i0 < n)
#pragma unroll 4
            for (int q = q0; q < jc; ++q) {
                const double4_32a p = s_j[q].f;
                const double dx = p.x - pi.x, dy = p.y - pi.y, dz = p.z - pi.z;
                const double y = rsqrt_pair(fma(dx, dx, fma(dy, dy, fma(dz, dz, eps2))));
                // i < j holds off the diagonal (lanes past the end are dropped
                // below); a pair left out may be infinite, so its term is not formed
                if (j0 + q > i) row = fma(p.w, y, row);
            }
    }
    row = i < n ? pi.w * row : 0.0;   // a particle past the end
#pragma unroll
    for (int off = 16; off >= 1; off >>= 1) row += __shfl_xor_sync(0xffffffffu, row, off);
    if (lane == 0) s_red[warp] = row;
    __syncthreads();
    if (tid == 0) part[blockIdx.x] = -((s_red[0] + s_red[1]) + (s_red[2] + s_red[3]));
}

// Kinetic energies, and the sums of the clusters' tiles.
template <int NT>
__global__ void __launch_bounds__(NT) k_ens_energy(EnsArgs ea, const int *item, const double *part,
                                                   double *ekin, double *epot)
{
    __shared__ double s_red[NT / 32];
    const int tid = threadIdx.x;
    const State &S = ea.s;
    const long long P = S.n;
    for (int c = blockIdx.x; c < ea.C; c += gridDim.x) {
        const long long o = ea.off[c];
        const int n = (int)(ea.off[c + 1] - o);
        double ke = 0.0, pe = 0.0;
        for (int i = tid; i < n; i += NT) {
            const long long gi = o + i;
            const double vx = S.v[gi], vy = S.v[P + gi], vz = S.v[2 * P + gi];
            ke += 0.5 * S.m[gi] * (vx * vx + vy * vy + vz * vz);
        }
        for (int q = item[c] + tid; q < item[c + 1]; q += NT) pe += part[q];
        struct Add {
            __device__ double operator()(double a, double b) const { return a + b; }
        };
        ke = cta_reduce(ke, Add(), s_red);
        pe = cta_reduce(pe, Add(), s_red);
        if (tid == 0) {
            ekin[c] = ke;
            epot[c] = pe;
        }
    }
}

// host AoS [P][3] -> device SoA staging -> state arrays
__global__ void k_aos_to_soa(const double *aos, double *soa, long long P)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < 3 * P;
         e += (long long)gridDim.x * blockDim.x) {
        const long long i = e / 3, c = e % 3;
        soa[c * P + i] = aos[e];
    }
}

__global__ void k_soa_to_aos(const double *soa, double *aos, long long P)
{
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < 3 * P;
         e += (long long)gridDim.x * blockDim.x) {
        const long long i = e / 3, c = e % 3;
        aos[e] = soa[c * P + i];
    }
}

}  // namespace
}  // namespace nbk

using namespace nbk;

// ---------------------------------------------------------------------------
// Host side: the nb_ens context and its C ABI.

struct nb_ens {
    int C = 0;
    long long P = 0;
    double eps = 0.0;
    nb_opts o{};
    cudaStream_t st = nullptr;
    bool own_stream = false;
    int sms = 0;
    State S{};
    long long *d_off = nullptr;
    int *d_order = nullptr;
    double *d_x = nullptr, *d_v = nullptr, *d_a = nullptr, *d_k = nullptr, *d_m = nullptr;
    long long *d_t = nullptr;
    int *d_lev = nullptr;
    int *d_work = nullptr, *d_done = nullptr, *d_err = nullptr;  // d_work: [2 + kEnsClasses] counters
    float4 *d_jph = nullptr, *d_jpl = nullptr, *d_jv = nullptr;
    float4 *d_mirror = nullptr;  // [5 P]: x_hi + m, x_lo, v, a, k in single precision
    int *d_act = nullptr, *d_na = nullptr;
    int2 *d_queue = nullptr, *d_pitem = nullptr;
    int npitem = 0, qbase[kEnsClasses] = {};
    long long *d_tnext = nullptr;
    long long *d_steps = nullptr, *d_inter = nullptr;
    double *d_stage = nullptr;   // [7 P] host I/O staging
    int *d_item = nullptr;       // [C + 1] first pair tile of each cluster (energies)
    int items = 0;
    double *d_backup = nullptr;  // state copy for tuning
    long long *d_tbak = nullptr;
    int *d_lbak = nullptr;
    int nt = 256, gmax = 8;      // order of the sums (tunable): gmax lanes, blocks of min(64 gmax, nt) j
    long long t_end = LLONG_MAX;
    cudaGraphExec_t graph = nullptr, graph_n = nullptr;   // one step, kEnsGraphSteps of them
    int graph_nt = 0, graph_gmax = 0;
    long long graph_tend = -1;
    long long launches = 0;
    std::string err;
};

namespace ens_impl {

thread_local std::string g_ens_init_err;

// An NVTX range over one entry point (no cost unless a tool is attached).
struct EnsRange {
    explicit EnsRange(const char *name) { nvtxRangePushA(name); }
    ~EnsRange() { nvtxRangePop(); }
};

int efail(nb_ens *e, int code, const char *fmt, ...)
{
    if (e) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        e->err = buf;
    }
    return code;
}

#define ECK(call)                                                                         \
    do {                                                                                  \
        cudaError_t e_ = (call);                                                          \
        if (e_ != cudaSuccess)                                                            \
            return efail(e, e_ == cudaErrorMemoryAllocation ? NB_ENOMEM : NB_ECUDA,       \
                         "%s: %s", #call, cudaGetErrorString(e_));                        \
    } while (0)

EnsArgs ens_args(nb_ens *e)
{
    EnsArgs a{};
    a.C = e->C;
    a.off = e->d_off;
    a.order = e->d_order;
    a.s = e->S;
    a.eps2 = (float)(e->eps * e->eps);
    a.eta = e->o.eta;
    a.eta_init = e->o.eta_init;
    a.level_min = e->o.level_min;
    a.t_end = e->t_end;
    a.g = e->gmax;
    a.sb = std::min(64 * e->gmax, e->nt);
    a.work = e->d_work;
    a.queue = e->d_queue;
    a.pitem = e->d_pitem;
    for (int k = 0; k < kEnsClasses; ++k) a.qbase[k] = e->qbase[k];
    a.jph = e->d_jph;
    a.jpl = e->d_jpl;
    a.jv = e->d_jv;
    a.mir.h = e->d_mirror;
    a.mir.l = e->d_mirror + e->P;
    a.mir.v = e->d_mirror + 2 * e->P;
    a.mir.a = e->d_mirror + 3 * e->P;
    a.mir.k = e->d_mirror + 4 * e->P;
    a.act = e->d_act;
    a.na = e->d_na;
    a.tnext = e->d_tnext;
    a.done = e->d_done;
    a.steps = e->d_steps;
    a.inter = e->d_inter;
    a.err = e->d_err;
    return a;
}

// One pass: schedule (with the small clusters' prediction), prediction of the
// larger ones, force and correction.
template <int MODE>
int enqueue_ens(nb_ens *e, const EnsArgs &a)
{
    int bps = 0;
    const auto force = a.eps2 > 0.0f ? k_ens_force<MODE, true> : k_ens_force<MODE, false>;
    ECK(cudaOccupancyMaxActiveBlocksPerMultiprocessor(&bps, force, kEnsFNT, 0));
    k_ens_sched<MODE><<<e->C, kEnsANT, 0, e->st>>>(a);
    if (e->npitem) k_ens_predict<MODE><<<e->npitem, kEnsPNT, 0, e->st>>>(a);
    force<<<e->sms * std::max(1, bps), kEnsFNT, 0, e->st>>>(a);
    ECK(cudaGetLastError());
    e->launches += 1;
    return NB_OK;
}

// One ensemble block step.
int enqueue_ens_step(nb_ens *e) { return enqueue_ens<kEnsStep>(e, ens_args(e)); }

// Refreshes the single-precision mirror after the FP64 state was set from outside a step.
int enqueue_mirror(nb_ens *e)
{
    k_ens_mirror<<<(int)std::min<long long>(8LL * e->sms, (e->P + 255) / 256), 256, 0, e->st>>>(
        ens_args(e));
    ECK(cudaGetLastError());
    e->launches += 1;
    return NB_OK;
}

int ens_sync(nb_ens *e)
{
    int h_err = 0;
    ECK(cudaMemcpyAsync(&h_err, e->d_err, sizeof(int), cudaMemcpyDeviceToHost, e->st));
    ECK(cudaStreamSynchronize(e->st));
    ECK(cudaGetLastError());
    if (h_err) {
        ECK(cudaMemsetAsync(e->d_err, 0, sizeof(int), e->st));
        ECK(cudaStreamSynchronize(e->st));
        return efail(e, h_err, "a new time step fell below 2^-40 in some cluster");
    }
    return NB_OK;
}

template <typename T>
int ealloc(nb_ens *e, T **p, long long count)
{
    if (count < 1) count = 1;
    if (cudaMalloc((void **)p, sizeof(T) * (size_t)count) != cudaSuccess) {
        *p = nullptr;
        cudaGetLastError();
        return efail(e, NB_ENOMEM, "cudaMalloc of %lld bytes failed", (long long)(sizeof(T) * count));
    }
    return NB_OK;
}

void drop_graphs(nb_ens *e)
{
    if (e->graph) cudaGraphExecDestroy(e->graph);
    if (e->graph_n) cudaGraphExecDestroy(e->graph_n);
    e->graph = e->graph_n = nullptr;
}

// `steps` ensemble steps as one graph.
int capture_steps(nb_ens *e, int steps, cudaGraphExec_t *out)
{
    cudaGraph_t g;
    const long long l0 = e->launches;
    ECK(cudaStreamBeginCapture(e->st, cudaStreamCaptureModeThreadLocal));
    int rc = NB_OK;
    for (int q = 0; q < steps && !rc; ++q) rc = enqueue_ens_step(e);
    e->launches = l0;
    cudaError_t ce = cudaStreamEndCapture(e->st, &g);
    if (rc) {
        if (ce == cudaSuccess && g) cudaGraphDestroy(g);
        return rc;
    }
    if (ce != cudaSuccess) return efail(e, NB_ECUDA, "graph capture: %s", cudaGetErrorString(ce));
    ce = cudaGraphInstantiate(out, g, 0);
    cudaGraphDestroy(g);
    if (ce != cudaSuccess) {
        *out = nullptr;
        return efail(e, NB_ECUDA, "graph instantiate: %s", cudaGetErrorString(ce));
    }
    return NB_OK;
}

void ens_release(nb_ens *e)
{
    if (e->st) cudaStreamSynchronize(e->st);
    drop_graphs(e);
    void *ptrs[] = {e->d_off, e->d_order, e->d_x, e->d_v, e->d_a, e->d_k, e->d_m, e->d_t,
                    e->d_lev, e->d_work, e->d_done, e->d_err, e->d_steps, e->d_inter,
                    e->d_stage, e->d_backup, e->d_tbak, e->d_lbak, e->d_jph, e->d_jpl, e->d_jv,
                    e->d_mirror,
                    e->d_act, e->d_na, e->d_queue, e->d_pitem, e->d_tnext, e->d_item};
    for (void *p : ptrs)
        if (p) cudaFree(p);
    if (e->own_stream && e->st) cudaStreamDestroy(e->st);
}

bool finite_all(const double *p, long long cnt)
{
    for (long long i = 0; i < cnt; ++i)
        if (!std::isfinite(p[i])) return false;
    return true;
}

int grid_of(long long n) { return (int)std::min<long long>(4096, std::max<long long>(1, (n + 255) / 256)); }

int ens_init_impl(nb_ens *e, int32_t C, const int64_t *off, const double *m, const double *x,
                  const double *v, double eps, const nb_opts *opts)
{
    nb_opts o;
    nb_default_opts(&o);
    if (opts) o = *opts;
    if (C < 1 || !off || !m || !x || !v) return efail(e, NB_EINVAL, "bad arguments");
    if (!std::isfinite(eps) || eps < 0.0) return efail(e, NB_EINVAL, "eps must be finite and >= 0");
    if (o.level_min < 0 || o.level_min > kTickBits || o.level_fixed != 0 || o.precision != NB_DS)
        return efail(e, NB_EINVAL, "ensembles use DS precision and individual block steps");
    if (o.summation != NB_SUM_COMPENSATED)
        return efail(e, NB_EINVAL, "ensembles use the compensated summation");
    if (!(o.eta > 0.0) || !(o.eta_init > 0.0)) return efail(e, NB_EINVAL, "eta must be positive");
    if (off[0] != 0) return efail(e, NB_EINVAL, "offsets must start at 0");
    std::vector<std::pair<long long, int>> sizes;
    for (int c = 0; c < C; ++c) {
        const long long nc = off[c + 1] - off[c];
        if (nc < 1 || nc > kEnsMaxN)
            return efail(e, NB_EINVAL, "cluster %d has %lld particles (1..%d allowed)", c, nc, kEnsMaxN);
        sizes.push_back({-nc, c});
    }
    const long long P = off[C];
    if (P > INT_MAX / 8) return efail(e, NB_EINVAL, "too many particles");
    if (!finite_all(m, P) || !finite_all(x, 3 * P) || !finite_all(v, 3 * P))
        return efail(e, NB_EINVAL, "non-finite input");
    for (long long i = 0; i < P; ++i)
        if (m[i] < 0.0) return efail(e, NB_EINVAL, "negative mass");
    std::stable_sort(sizes.begin(), sizes.end());
    std::vector<int> order(C);
    // a cluster has at most n force items: the classes' parts of the queue
    std::vector<int2> pitem;
    for (int q = 0; q < C; ++q) {
        const int c = order[q] = sizes[q].second, nc = (int)-sizes[q].first;
        for (int k = ens_class(nc) + 1; k < kEnsClasses; ++k) e->qbase[k] += nc;
        if (nc > kEnsPredChunk)
            for (int p = 0; p * kEnsPredChunk < nc; ++p) pitem.push_back(make_int2(c, p));
    }
    e->npitem = (int)pitem.size();

    e->C = C;
    e->P = P;
    e->eps = eps;
    e->o = o;
    if (o.stream) {
        e->st = (cudaStream_t)o.stream;
    } else {
        ECK(cudaStreamCreateWithFlags(&e->st, cudaStreamNonBlocking));
        e->own_stream = true;
    }
    int dev = 0;
    ECK(cudaGetDevice(&dev));
    ECK(cudaDeviceGetAttribute(&e->sms, cudaDevAttrMultiProcessorCount, dev));
    int rc;
    if ((rc = ealloc(e, &e->d_off, C + 1)) || (rc = ealloc(e, &e->d_order, C)) ||
        (rc = ealloc(e, &e->d_x, 3 * P)) || (rc = ealloc(e, &e->d_v, 3 * P)) ||
        (rc = ealloc(e, &e->d_a, 3 * P)) || (rc = ealloc(e, &e->d_k, 3 * P)) ||
        (rc = ealloc(e, &e->d_m, P)) || (rc = ealloc(e, &e->d_t, P)) || (rc = ealloc(e, &e->d_lev, P)) ||
        (rc = ealloc(e, &e->d_work, 2 + kEnsClasses)) || (rc = ealloc(e, &e->d_done, C)) || (rc = ealloc(e, &e->d_err, 1)) ||
        (rc = ealloc(e, &e->d_steps, C)) || (rc = ealloc(e, &e->d_inter, C)) ||
        (rc = ealloc(e, &e->d_stage, 7 * P)) || (rc = ealloc(e, &e->d_jph, P)) ||
        (rc = ealloc(e, &e->d_jpl, P)) || (rc = ealloc(e, &e->d_jv, P)) ||
        (rc = ealloc(e, &e->d_act, P)) || (rc = ealloc(e, &e->d_na, C)) ||
        (rc = ealloc(e, &e->d_tnext, C)) || (rc = ealloc(e, &e->d_queue, P)) ||
        (rc = ealloc(e, &e->d_pitem, std::max<long long>(1, (long long)pitem.size()))) ||
        (rc = ealloc(e, &e->d_mirror, 5 * P)) || (rc = ealloc(e, &e->d_item, C + 1)))
        return rc;
    // at most one tile per particle, so the tile sums fit the staging buffer
    std::vector<int> item(C + 1, 0);
    for (int c = 0; c < C; ++c) item[c + 1] = item[c] + (int)en_items((int)(off[c + 1] - off[c]));
    e->items = item[C];
    e->S.x = e->d_x;
    e->S.v = e->d_v;
    e->S.a = e->d_a;
    e->S.k = e->d_k;
    e->S.m = e->d_m;
    e->S.t = e->d_t;
    e->S.lev = e->d_lev;
    e->S.n = (int)P;
    ECK(cudaMemcpyAsync(e->d_off, off, sizeof(long long) * (C + 1), cudaMemcpyHostToDevice, e->st));
    ECK(cudaMemcpyAsync(e->d_order, order.data(), sizeof(int) * C, cudaMemcpyHostToDevice, e->st));
    ECK(cudaMemcpyAsync(e->d_item, item.data(), sizeof(int) * (C + 1), cudaMemcpyHostToDevice, e->st));
    ECK(cudaMemcpyAsync(e->d_m, m, sizeof(double) * P, cudaMemcpyHostToDevice, e->st));
    ECK(cudaMemcpyAsync(e->d_stage, x, sizeof(double) * 3 * P, cudaMemcpyHostToDevice, e->st));
    k_aos_to_soa<<<grid_of(3 * P), 256, 0, e->st>>>(e->d_stage, e->d_x, P);
    ECK(cudaStreamSynchronize(e->st));
    ECK(cudaMemcpyAsync(e->d_stage, v, sizeof(double) * 3 * P, cudaMemcpyHostToDevice, e->st));
    k_aos_to_soa<<<grid_of(3 * P), 256, 0, e->st>>>(e->d_stage, e->d_v, P);
    ECK(cudaMemsetAsync(e->d_a, 0, sizeof(double) * 3 * P, e->st));
    ECK(cudaMemsetAsync(e->d_k, 0, sizeof(double) * 3 * P, e->st));
    ECK(cudaMemsetAsync(e->d_t, 0, sizeof(long long) * P, e->st));
    ECK(cudaMemsetAsync(e->d_done, 0, sizeof(int) * C, e->st));
    ECK(cudaMemsetAsync(e->d_err, 0, sizeof(int), e->st));
    ECK(cudaMemsetAsync(e->d_steps, 0, sizeof(long long) * C, e->st));
    ECK(cudaMemsetAsync(e->d_inter, 0, sizeof(long long) * C, e->st));
    if (!pitem.empty())
        ECK(cudaMemcpyAsync(e->d_pitem, pitem.data(), sizeof(int2) * pitem.size(), cudaMemcpyHostToDevice, e->st));
    ECK(cudaMemsetAsync(e->d_work, 0, sizeof(int) * (2 + kEnsClasses), e->st));
    // start-up: force on every particle of every cluster, initial steps
    if ((rc = enqueue_ens<kEnsInit>(e, ens_args(e)))) return rc;
    ECK(cudaGetLastError());
    if ((rc = enqueue_mirror(e))) return rc;
    return ens_sync(e);
}

}  // namespace ens_impl

using namespace ens_impl;

extern "C" {

int nb_ens_init(nb_ens **ens, int32_t n_clusters, const int64_t *offsets, const double *m,
                const double *x, const double *v, double eps, const nb_opts *opts)
{
    const EnsRange range_("nb_ens_init");
    g_ens_init_err.clear();
    if (!ens) return NB_EINVAL;
    *ens = nullptr;
    nb_ens *e = new (std::nothrow) nb_ens();
    if (!e) return NB_ENOMEM;
    const int rc = ens_init_impl(e, n_clusters, offsets, m, x, v, eps, opts);
    if (rc != NB_OK) {
        g_ens_init_err = e->err;
        ens_release(e);
        delete e;
        return rc;
    }
    *ens = e;
    return NB_OK;
}

void nb_ens_free(nb_ens *e)
{
    if (!e) return;
    ens_release(e);
    delete e;
}

const char *nb_ens_last_error(const nb_ens *e)
{
    if (e) return e->err.c_str();
    return g_ens_init_err.empty() ? "null ensemble" : g_ens_init_err.c_str();
}

int nb_ens_configure(nb_ens *e, int threads, int gmax)
{
    if (!e) return NB_EINVAL;
    if ((threads != 128 && threads != 256 && threads != 512) ||
        (gmax != 1 && gmax != 2 && gmax != 4 && gmax != 8 && gmax != 16 && gmax != 32))
        return efail(e, NB_EINVAL, "threads in {128, 256, 512}, gmax a power of two <= 32");
    e->nt = threads;
    e->gmax = gmax;
    return NB_OK;
}

int nb_ens_run(nb_ens *e, double t_end, int64_t max_launches, int64_t *launches_out,
               int64_t *interactions_out)
{
    const EnsRange range_("nb_ens_run");
    if (!e) return NB_EINVAL;
    if (!std::isfinite(t_end) || t_end < 0.0 || t_end >= 0x1p22 || t_end * 0x1p40 != std::floor(t_end * 0x1p40))
        return efail(e, NB_EINVAL, "t_end is not on the 2^-40 grid");
    if (max_launches < 0) return efail(e, NB_EINVAL, "max_launches < 0");
    const long long te = (long long)(t_end * 0x1p40);
    if (te != e->t_end) {
        // a new end time re-opens finished clusters
        ECK(cudaMemsetAsync(e->d_done, 0, sizeof(int) * e->C, e->st));
        e->t_end = te;
    }
    // one ensemble step, and a stretch of them (a graph's start costs about 5 us), as graphs
    if (!e->graph || e->graph_nt != e->nt || e->graph_gmax != e->gmax || e->graph_tend != te) {
        drop_graphs(e);
        const int rc = capture_steps(e, 1, &e->graph);
        if (rc) return rc;
        e->graph_nt = e->nt;
        e->graph_gmax = e->gmax;
        e->graph_tend = te;
    }
    std::vector<int> done(e->C);
    long long n = 0;
    std::vector<long long> inter0(e->C), inter1(e->C);
    ECK(cudaMemcpyAsync(inter0.data(), e->d_inter, sizeof(long long) * e->C, cudaMemcpyDeviceToHost, e->st));
    while (n < max_launches) {
        const long long k = std::min<long long>(32, max_launches - n);
        long long q = 0;
        if (k == 32) {   // a longer graph only where its capture pays
            const int rc = e->graph_n ? NB_OK : capture_steps(e, kEnsGraphSteps, &e->graph_n);
            if (rc) return rc;
            for (; q < k; q += kEnsGraphSteps) ECK(cudaGraphLaunch(e->graph_n, e->st));
        }
        for (; q < k; ++q) ECK(cudaGraphLaunch(e->graph, e->st));
        n += k;
        e->launches += k;
        ECK(cudaMemcpyAsync(done.data(), e->d_done, sizeof(int) * e->C, cudaMemcpyDeviceToHost, e->st));
        int rc = ens_sync(e);
        if (rc) return rc;
        bool all = true;
        for (int c = 0; c < e->C && all; ++c) all = done[c] != 0;
        if (all) break;
    }
    ECK(cudaMemcpyAsync(inter1.data(), e->d_inter, sizeof(long long) * e->C, cudaMemcpyDeviceToHost, e->st));
    ECK(cudaStreamSynchronize(e->st));
    long long it = 0;
    for (int c = 0; c < e->C; ++c) it += inter1[c] - inter0[c];
    if (launches_out) *launches_out = n;
    if (interactions_out) *interactions_out = it;
    return NB_OK;
}

int nb_ens_tune(nb_ens *e, int launches_per_candidate, int *threads_out, int *gmax_out,
                double *ms_out)
{
    const EnsRange range_("nb_ens_tune");
    if (!e) return NB_EINVAL;
    if (launches_per_candidate < 1) return efail(e, NB_EINVAL, "launches_per_candidate < 1");
    const long long P = e->P, C = e->C;
    int rc;
    if (!e->d_backup && ((rc = ealloc(e, &e->d_backup, 12 * P + 2 * C)) ||
                         (rc = ealloc(e, &e->d_tbak, P)) || (rc = ealloc(e, &e->d_lbak, P + C))))
        return rc;
    // snapshot: x, v, a, k, times, levels, per-cluster counters and flags
    double *arrs[4] = {e->d_x, e->d_v, e->d_a, e->d_k};
    auto save = [&](bool restore) -> int {
        for (int q = 0; q < 4; ++q) {
            double *b = e->d_backup + q * 3 * P;
            ECK(cudaMemcpyAsync(restore ? arrs[q] : b, restore ? b : arrs[q], sizeof(double) * 3 * P,
                                cudaMemcpyDeviceToDevice, e->st));
        }
        long long *cb = (long long *)(e->d_backup + 12 * P);
        ECK(cudaMemcpyAsync(restore ? e->d_t : e->d_tbak, restore ? e->d_tbak : e->d_t,
                            sizeof(long long) * P, cudaMemcpyDeviceToDevice, e->st));
        ECK(cudaMemcpyAsync(restore ? e->d_lev : e->d_lbak, restore ? e->d_lbak : e->d_lev,
                            sizeof(int) * P, cudaMemcpyDeviceToDevice, e->st));
        ECK(cudaMemcpyAsync(restore ? e->d_done : e->d_lbak + P, restore ? e->d_lbak + P : e->d_done,
                            sizeof(int) * C, cudaMemcpyDeviceToDevice, e->st));
        ECK(cudaMemcpyAsync(restore ? e->d_steps : cb, restore ? cb : e->d_steps,
                            sizeof(long long) * C, cudaMemcpyDeviceToDevice, e->st));
        ECK(cudaMemcpyAsync(restore ? e->d_inter : cb + C, restore ? cb + C : e->d_inter,
                            sizeof(long long) * C, cudaMemcpyDeviceToDevice, e->st));
        return restore ? enqueue_mirror(e) : NB_OK;
    };
    if ((rc = save(false))) return rc;
    cudaEvent_t e0, e1;
    ECK(cudaEventCreate(&e0));
    ECK(cudaEventCreate(&e1));
    const int cand_nt[3] = {128, 256, 512};
    const int cand_g[6] = {1, 2, 4, 8, 16, 32};
    float best = 1e30f;
    int bnt = e->nt, bg = e->gmax;
    for (int a = 0; a < 3; ++a)
        for (int b = 0; b < 6; ++b) {
            e->nt = cand_nt[a];
            e->gmax = cand_g[b];
            if ((rc = save(true))) return rc;
            if ((rc = enqueue_ens_step(e))) return rc;  // warm-up
            ECK(cudaEventRecord(e0, e->st));
            for (int q = 0; q < launches_per_candidate; ++q)
                if ((rc = enqueue_ens_step(e))) return rc;
            ECK(cudaEventRecord(e1, e->st));
            if ((rc = ens_sync(e))) return rc;
            float ms = 0.0f;
            ECK(cudaEventElapsedTime(&ms, e0, e1));
            if (ms < best) {
                best = ms;
                bnt = e->nt;
                bg = e->gmax;
            }
        }
    cudaEventDestroy(e0);
    cudaEventDestroy(e1);
    if ((rc = save(true))) return rc;
    ECK(cudaStreamSynchronize(e->st));
    e->nt = bnt;
    e->gmax = bg;
    if (threads_out) *threads_out = bnt;
    if (gmax_out) *gmax_out = bg;
    if (ms_out) *ms_out = best / launches_per_candidate;
    return NB_OK;
}

int nb_ens_step(nb_ens *e)
{
    const EnsRange range_("nb_ens_step");
    if (!e) return NB_EINVAL;
    int rc = enqueue_ens_step(e);
    if (rc) return rc;
    return ens_sync(e);
}

int nb_ens_force(nb_ens *e, double *acc, double *jerk, double *pot)
{
    const EnsRange range_("nb_ens_force");
    if (!e) return NB_EINVAL;
    const long long P = e->P;
    EnsArgs a = ens_args(e);
    a.out_acc = e->d_stage;
    a.out_jerk = e->d_stage + 3 * P;
    a.out_pot = e->d_stage + 6 * P;
    int rc = enqueue_ens<kEnsForce>(e, a);
    if (rc) return rc;
    if (acc) ECK(cudaMemcpyAsync(acc, a.out_acc, sizeof(double) * 3 * P, cudaMemcpyDeviceToHost, e->st));
    if (jerk) ECK(cudaMemcpyAsync(jerk, a.out_jerk, sizeof(double) * 3 * P, cudaMemcpyDeviceToHost, e->st));
    if (pot) ECK(cudaMemcpyAsync(pot, a.out_pot, sizeof(double) * P, cudaMemcpyDeviceToHost, e->st));
    return ens_sync(e);
}

int nb_ens_energy(nb_ens *e, double *ekin, double *epot)
{
    const EnsRange range_("nb_ens_energy");
    if (!e) return NB_EINVAL;
    double *d = e->d_stage;
    double *part = d + 2LL * e->C;
    k_ens_pairs<<<e->items, kEnTile, 0, e->st>>>(ens_args(e), e->d_item, e->eps * e->eps, part);
    k_ens_energy<256><<<std::max(1, std::min(e->C, 8 * e->sms)), 256, 0, e->st>>>(
        ens_args(e), e->d_item, part, d, d + e->C);
    ECK(cudaGetLastError());
    e->launches += 2;
    if (ekin) ECK(cudaMemcpyAsync(ekin, d, sizeof(double) * e->C, cudaMemcpyDeviceToHost, e->st));
    if (epot) ECK(cudaMemcpyAsync(epot, d + e->C, sizeof(double) * e->C, cudaMemcpyDeviceToHost, e->st));
    return ens_sync(e);
}

int nb_ens_get_state(nb_ens *e, double *x, double *v, double *a, double *k, int64_t *t,
                     int32_t *level, int64_t *steps, int64_t *interactions)
{
    if (!e) return NB_EINVAL;
    const long long P = e->P;
    double *src[4] = {e->d_x, e->d_v, e->d_a, e->d_k};
    double *dst[4] = {x, v, a, k};
    for (int q = 0; q < 4; ++q) {
        if (!dst[q]) continue;
        k_soa_to_aos<<<grid_of(3 * P), 256, 0, e->st>>>(src[q], e->d_stage, P);
        ECK(cudaMemcpyAsync(dst[q], e->d_stage, sizeof(double) * 3 * P, cudaMemcpyDeviceToHost, e->st));
        ECK(cudaStreamSynchronize(e->st));
    }
    if (t) ECK(cudaMemcpyAsync(t, e->d_t, sizeof(long long) * P, cudaMemcpyDeviceToHost, e->st));
    if (level) ECK(cudaMemcpyAsync(level, e->d_lev, sizeof(int) * P, cudaMemcpyDeviceToHost, e->st));
    if (steps) ECK(cudaMemcpyAsync(steps, e->d_steps, sizeof(long long) * e->C, cudaMemcpyDeviceToHost, e->st));
    if (interactions)
        ECK(cudaMemcpyAsync(interactions, e->d_inter, sizeof(long long) * e->C, cudaMemcpyDeviceToHost, e->st));
    return ens_sync(e);
}

int nb_ens_set_state(nb_ens *e, const double *x, const double *v, const double *a, const double *k,
                     const int64_t *t, const int32_t *level)
{
    if (!e) return NB_EINVAL;
    if (!x || !v || !a || !k || !t || !level) return efail(e, NB_EINVAL, "all arrays are required");
    const long long P = e->P;
    if (!finite_all(x, 3 * P) || !finite_all(v, 3 * P) || !finite_all(a, 3 * P) || !finite_all(k, 3 * P))
        return efail(e, NB_EINVAL, "non-finite state");
    for (long long i = 0; i < P; ++i) {
        if (level[i] < e->o.level_min || level[i] > kTickBits) return efail(e, NB_EINVAL, "bad level");
        if (t[i] < 0 || t[i] % (1LL << (kTickBits - level[i])) != 0)
            return efail(e, NB_EINVAL, "time not a multiple of its step");
    }
    const double *src[4] = {x, v, a, k};
    double *dst[4] = {e->d_x, e->d_v, e->d_a, e->d_k};
    for (int q = 0; q < 4; ++q) {
        ECK(cudaMemcpyAsync(e->d_stage, src[q], sizeof(double) * 3 * P, cudaMemcpyHostToDevice, e->st));
        k_aos_to_soa<<<grid_of(3 * P), 256, 0, e->st>>>(e->d_stage, dst[q], P);
        ECK(cudaStreamSynchronize(e->st));
    }
    ECK(cudaMemcpyAsync(e->d_t, t, sizeof(long long) * P, cudaMemcpyHostToDevice, e->st));
    ECK(cudaMemcpyAsync(e->d_lev, level, sizeof(int) * P, cudaMemcpyHostToDevice, e->st));
    ECK(cudaMemsetAsync(e->d_done, 0, sizeof(int) * e->C, e->st));
    int rc = enqueue_mirror(e);
    if (rc) return rc;
    return ens_sync(e);
}

}  // extern "C"
