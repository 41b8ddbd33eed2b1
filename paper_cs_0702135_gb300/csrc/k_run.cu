// k_run.cu -- the block-step loop of nb_run (Section 2: select the block,
// predict, force, correct, repeat) in one persistent cooperative launch, for
// systems small enough that a step is mostly launch latency on the
// kernel-per-stage path.
//
// CTA r owns particles [r P, (r + 1) P) and keeps their whole state in shared
// memory for the length of the launch.  One block step:
//   1. the CTA corrects its own particles of the previous block: a warp adds a
//      particle's partials over the CTAs (lanes over CTAs, then a fixed
//      reduce-scatter tree), then the FP64 corrector and Aarseth step run (four
//      lanes per particle for up to 16 particles); the least end time
//      t_i + 2^-lev_i of its particles and how many end then are published;
//   2. from all CTAs' published pairs the block time t_next, the block size and
//      the CTA's offset in the block (the same in every CTA, so every CTA takes
//      the same decision to stop); its particles predicted (FP64) into
//      double-single j records in shared memory, those of its block members
//      published at their block positions (fixed point: also its largest mass
//      and |vx|+|vy|+|vz|);
//   3. force partials: every CTA sums every block particle's pair terms over
//      its own particles as j and writes them per (block particle, CTA), then
//      raises its step flag.
//
// No grid barrier: each exchange is a 16-byte record that carries its step
// (128-bit relaxed accesses are single transactions), so the reader that finds
// the step's tag has the data with it; only the partials, which are longer, sit
// behind a release flag.  A record is overwritten one exchange later at the
// earliest: a CTA publishes its end time of step s + 1 only after its force of
// step s, block records of s + 1 follow from all CTAs' end times of s + 1, and
// partials of s + 1 from those; the end times themselves alternate between two
// slots, because a CTA without block particles may still be reading step s
// when another publishes s + 1.  Every wait ends after about 2 s with
// NB_ETIMEOUT, and the cooperative launch keeps every CTA resident.
//
// Bound by latency: at N = 1024 a step was 36,000 clocks with the state in
// global memory and three grid barriers (waits at barriers 15,000, force 6,500,
// prediction 3,700, block list 3,600, partial sums 3,500, corrector 2,900),
// 19.2 us a step with the copies around the run; now 10.5 us (18.5 then, counted the
// same way: 1/8 time unit with nb_set_state before it).
//
// Two summations: the compensated double-single sums (TwoSum-promoted FP32
// partials, FP64 across CTAs) and the GRAPE-style fixed-point sums of k_sum.cu
// (exact, so the run is bit-identical to the kernel-per-stage path and to any
// IEEE evaluation of the same sums).
#include <climits>

#include "nb_device.cuh"

namespace nbk {
namespace {

using namespace dev;

constexpr unsigned kFullR = 0xffffffffu;
constexpr long long kRunSpinCycles = 4000000000LL;  // about 2 s at 2 GHz

__device__ __forceinline__ void store_release(unsigned long long *p, unsigned long long v)
{
    asm volatile("st.release.gpu.global.u64 [%0], %1;" ::"l"(p), "l"(v) : "memory");
}

// 16 bytes in one access, past L1.
__device__ __forceinline__ void store128(void *p, ulonglong2 v)
{
    asm volatile("{\n\t.reg .b128 q;\n\tmov.b128 q, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], q;\n\t}" ::"l"(p),
                 "l"(v.x), "l"(v.y)
                 : "memory");
}
__device__ __forceinline__ ulonglong2 load128(const void *p)
{
    ulonglong2 v;
    asm volatile("{\n\t.reg .b128 q;\n\tld.relaxed.gpu.global.b128 q, [%2];\n\tmov.b128 {%0, %1}, q;\n\t}"
                 : "=l"(v.x), "=l"(v.y)
                 : "l"(p)
                 : "memory");
    return v;
}
__device__ __forceinline__ unsigned tag_of(ulonglong2 v) { return (unsigned)(v.y >> 32); }

__device__ __forceinline__ unsigned long long load_acquire(const unsigned long long *p)
{
    unsigned long long v;
    asm volatile("ld.acquire.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}

// Bounded wait (one thread): until *p >= target, read with acquire semantics;
// false after `limit` SM cycles.  Spins first, then sleeps between reads.
__device__ __forceinline__ bool wait_counter(const unsigned long long *p, unsigned long long target,
                                             long long limit)
{
    const long long t0 = clock64();
    int spins = 0;
    while (load_acquire(p) < target) {
        if (++spins > 256) {
            if (clock64() - t0 > limit) return false;
            __nanosleep(64);
        }
    }
    return true;
}

// The least of the lanes' non-negative values, by its two halves.
__device__ __forceinline__ long long warp_min(long long v)
{
    const unsigned hi = (unsigned)(v >> 32), mh = __reduce_min_sync(kFullR, hi);
    const unsigned ml = __reduce_min_sync(kFullR, hi == mh ? (unsigned)v : 0xffffffffu);
    return (long long)((unsigned long long)mh << 32 | ml);
}

// The limit of a wait that polls records or flags: false once it has run out.
struct Patience {
    long long t0 = 0;
    int spins = 0;
    __device__ __forceinline__ bool more()
    {
        if (++spins < 256) return true;
        if (spins == 256) t0 = clock64();
        if (clock64() - t0 > kRunSpinCycles) return false;
        __nanosleep(32);
        return true;
    }
};

// The same wait on a counter that nothing increments, for nb_check_wait.
__global__ void k_check_wait(const unsigned long long *counter, long long limit, Ctrl *ctrl)
{
    if (!wait_counter(counter, 1ULL, limit)) atomicCAS(&ctrl->err, 0, NB_ETIMEOUT);
}

// Lane l of the warp ends with the sum over the lanes of value l >> 2 (8
// values), added as the xor tree 16, 8, 4, 2, 1 adds each.
template <typename T, typename Add>
__device__ __forceinline__ T warp_scatter8(T (&v)[8], int lane, Add add)
{
#pragma unroll
    for (int lev = 0; lev < 3; ++lev) {
        const int off = 16 >> lev, half = 4 >> lev;
        const bool up = (lane & off) != 0;
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k < half) {
                const T send = up ? v[k] : v[k + half], keep = up ? v[k + half] : v[k];
                v[k] = add(keep, send, off);
            }
    }
    v[0] = add(v[0], v[0], 2);
    v[0] = add(v[0], v[0], 1);
    return v[0];
}

// add(keep, send, off): keep + the partner's send.
struct AddF64 {
    __device__ double operator()(double keep, double send, int off) const
    {
        return keep + __shfl_xor_sync(kFullR, send, off);
    }
};
struct Int128 {
    long long hi;
    unsigned long long lo;
};
struct AddI128 {
    __device__ Int128 operator()(Int128 k, Int128 s, int off) const
    {
        const long long h2 = __shfl_xor_sync(kFullR, s.hi, off);
        const unsigned long long l2 = __shfl_xor_sync(kFullR, s.lo, off);
        const unsigned long long ls = k.lo + l2;
        return {k.hi + h2 + (ls < k.lo ? 1 : 0), ls};
    }
};
struct DSVal {
    float h, l;
};
struct AddDS {
    __device__ DSVal operator()(DSVal k, DSVal s, int off) const
    {
        const float h2 = __shfl_xor_sync(kFullR, s.h, off), l2 = __shfl_xor_sync(kFullR, s.l, off);
        ds_add(k.h, k.l, h2, l2);
        return k;
    }
};

// The sums over a group of G consecutive lanes of 8 values each, added as the
// xor tree 1, 2, 4, ... adds them; lane q of the group (q < 8) keeps the
// values from `first` on, 8 / min(G, 8) of them.
template <int G, typename T, typename Add>
__device__ __forceinline__ void group_scatter8(T (&v)[8], int q, Add add, int &first)
{
    first = 0;
#pragma unroll
    for (int lev = 0; (1 << lev) < G; ++lev) {
        const int off = 1 << lev, half = 4 >> lev;
        if (half >= 1) {
            const bool up = (q & off) != 0;
#pragma unroll
            for (int k = 0; k < 4; ++k)
                if (k < half) {
                    const T send = up ? v[k] : v[k + half], keep = up ? v[k + half] : v[k];
                    v[k] = add(keep, send, off);
                }
            first += up ? half : 0;
        } else {
            v[0] = add(v[0], v[0], off);
        }
    }
}

// Record of block particle a at this step (waits for it): the particle's index,
// or -1 when the wait ran out.
__device__ __forceinline__ int block_record(const RunArgs &ra, int a, unsigned epoch, float4 &p, float4 &l, float4 &v)
{
    const float4 *src = ra.blk + 3 * (long long)a;
    Patience w;
    for (;;) {
        const ulonglong2 q0 = load128(src), q1 = load128(src + 1), q2 = load128(src + 2);
        const unsigned t0 = tag_of(q0), t1 = tag_of(q1), t2 = tag_of(q2);
        if (t0 >> kRunIndexBits == epoch && t1 == t0 && t2 == t0) {
            auto f = [](unsigned long long u, int k) { return __uint_as_float((unsigned)(u >> (32 * k))); };
            p = make_float4(f(q0.x, 0), f(q0.x, 1), f(q0.y, 0), 0.0f);
            l = make_float4(f(q1.x, 0), f(q1.x, 1), f(q1.y, 0), 0.0f);
            v = make_float4(f(q2.x, 0), f(q2.x, 1), f(q2.y, 0), 0.0f);
            return (int)(t0 & ((1u << kRunIndexBits) - 1u));
        }
        if (!w.more()) return -1;
    }
}

// Phase 3: block particles a in passes of NT / G, G lanes per particle
// splitting the CTA's j.  Compensated: FP32 partials promoted by TwoSum every
// 64 pairs per lane, the lane group reduced in double-single.  Fixed point:
// every term rounded to an integer by the exact FP32 splits, tiles of at most
// 64 terms per lane summed in 32 bits and then in 128 bits, the lane group
// reduced in 128 bits.  False when a wait ran out.
template <int MODE, int G>
__device__ __forceinline__ bool force_phase(const RunArgs &ra, int r, int na, int j0, int m, unsigned epoch,
                                            const float4 *s_p, const float4 *s_l, const float4 *s_v,
                                            const Scale &S)
{
    const int tid = threadIdx.x;
    const int grp = tid / G, lig = tid % G;
    bool ok = true;
    for (int a0 = 0; a0 < na; a0 += kRunNT / G) {
        const int a = a0 + grp;
        const bool valid = a < na;
        float4 ip, il, iv;
        const int i = block_record(ra, valid ? a : na - 1, epoch, ip, il, iv);
        if (i < 0) {
            ok = false;
            ip = il = iv = make_float4(0.f, 0.f, 0.f, 0.f);
        }
        double *const dst = ra.part + ((long long)a * ra.ncta + r) * (MODE == NB_SUM_FIXED ? 16 : 8);
        int first;
        constexpr int kKeep = G >= 8 ? 1 : 8 / G;
        if (MODE == NB_SUM_FIXED) {
            const float xh[3] = {ip.x, ip.y, ip.z}, xl[3] = {il.x, il.y, il.z}, vi[3] = {iv.x, iv.y, iv.z};
            Int128 t8[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) t8[c] = {0, 0};
            for (int jb = 0; jb < m; jb += 64 * G) {
                const int je = min(m, jb + 64 * G);
                unsigned s1[7], s2[7], s3[7];
#pragma unroll
                for (int c = 0; c < 7; ++c) s1[c] = s2[c] = s3[c] = 0u;
                unsigned cnt = 0;
                for (int jj = jb + lig; jj < je; jj += G) {
                    float t[7];
                    pair_rn(s_p[jj], s_l[jj], s_v[jj], xh, xl, vi, ra.eps2f, S.sc[0], S.sc[1], S.sc[2], t);
                    const bool self = j0 + jj == i;
#pragma unroll
                    for (int c = 0; c < 7; ++c) split_add(self ? 0.0f : t[c], s1[c], s2[c], s3[c]);
                    ++cnt;
                }
#pragma unroll
                for (int c = 0; c < 7; ++c) add128(t8[c].hi, t8[c].lo, tile_sum(s1[c], s2[c], s3[c], cnt));
            }
            group_scatter8<G>(t8, lig, AddI128(), first);
            if (valid && lig < 8)
#pragma unroll
                for (int k = 0; k < kKeep; ++k)
                    if (first + k < kComp) {
                        long long *p = reinterpret_cast<long long *>(dst) + 2 * (first + k);
                        p[0] = t8[k].hi;
                        p[1] = (long long)t8[k].lo;
                    }
        } else {
            const IDS I = make_ids(ip, il, iv);
            DSVal t8[8];
#pragma unroll
            for (int c = 0; c < 8; ++c) t8[c] = {0.0f, 0.0f};
            for (int jb = 0; jb < m; jb += 64 * G) {
                const int je = min(m, jb + 64 * G);
                float ta[3] = {0, 0, 0}, tk[3] = {0, 0, 0}, tp = 0.0f;
                for (int jj = jb + lig; jj < je; jj += G)
                    pair_ds_packed<false, true>(s_p[jj], s_l[jj], s_v[jj], I, ra.eps2f, ta, tk, tp,
                                                j0 + jj, i);
                const float t7[7] = {ta[0], ta[1], ta[2], tk[0], tk[1], tk[2], tp};
#pragma unroll
                for (int c = 0; c < 7; ++c) two_sum_acc(t8[c].h, t8[c].l, t7[c]);
            }
            group_scatter8<G>(t8, lig, AddDS(), first);
            if (valid && lig < 8)
#pragma unroll
                for (int k = 0; k < kKeep; ++k)
                    if (first + k < kComp) dst[first + k] = (double)t8[k].h + (double)t8[k].l;
        }
    }
    return ok;
}

// Bytes of shared memory per particle of a CTA (see k_run).
constexpr int kRunBytesPer = 12 * 8 + 8 + 8 + 8 * 8 + 3 * 16 + 4 + 4;

template <int MODE>
__global__ void __launch_bounds__(kRunNT) k_run(RunArgs ra)
{
    // this CTA's particles: state, end times, combined force of its block
    // members, j records
    extern __shared__ float4 s_dyn[];
    static_assert(alignof(decltype(s_dyn[0])) >= alignof(float4), "the records within need 16 bytes");
    const int per = ra.per;
    double *const s_st = reinterpret_cast<double *>(s_dyn);         // [12][per] x, v, a, k
    double *const s_res = s_st + 12 * per;                          // [per][8]
    float4 *const s_p = reinterpret_cast<float4 *>(s_res + 8 * per);
    float4 *const s_l = s_p + per, *const s_v = s_l + per;
    long long *const s_t = reinterpret_cast<long long *>(s_v + per);
    long long *const s_et = s_t + per;                              // t_i + 2^-lev_i
    int *const s_lev = reinterpret_cast<int *>(s_et + per);
    int *const s_blk = s_lev + per;                                 // block members (local indices)
    __shared__ long long s_tn;
    __shared__ int s_na, s_off, s_stop, s_err, s_late;
    __shared__ unsigned s_max[2][kRunNT / 32];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, r = blockIdx.x;
    const int n = ra.n, ncta = ra.ncta;
    const int i0 = r * per, i1 = min(n, i0 + per);
    const int m = max(0, i1 - i0);
    State L;   // the same particles as a State
    L.x = s_st, L.v = s_st + 3 * per, L.a = s_st + 6 * per, L.k = s_st + 9 * per;
    L.m = nullptr, L.t = s_t, L.lev = s_lev, L.n = per;

    if (tid < m) {
        const int i = i0 + tid;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            L.x[c * per + tid] = ra.s.x[(long long)c * n + i];
            L.v[c * per + tid] = ra.s.v[(long long)c * n + i];
            L.a[c * per + tid] = ra.s.a[(long long)c * n + i];
            L.k[c * per + tid] = ra.s.k[(long long)c * n + i];
        }
        s_t[tid] = ra.s.t[i];
        s_lev[tid] = ra.s.lev[i];
        s_et[tid] = s_t[tid] + (1LL << (kTickBits - s_lev[tid]));
        s_p[tid] = make_float4(0.0f, 0.0f, 0.0f, to_float_int(ra.s.m[i]));
        s_l[tid] = s_v[tid] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
    if (tid == 0) {
        s_err = ra.ctrl->err != 0;
        s_late = 0;
    }
    __syncthreads();
    long long steps = 0, inter = 0, tn_b = 0, tn_end = 0;
    int off_b = 0, cnt_b = 0, na_b = 0;
    bool past_end = false;
    Scale Sc;
    bool scale_ok = true;
    for (;;) {
        const unsigned epoch = (unsigned)(steps + 1);
        // 1. Own particles of the previous block (block positions off_b ..
        // off_b + cnt_b - 1): partials in CTA order, corrector, new steps.
        if (cnt_b > 0 && scale_ok) {
            if (warp < cnt_b) {
                // lane q adds the partials of CTAs q, q + 32, ...: it waits for
                // their flags of the step
                for (int q = lane; q < ncta; q += 32) {
                    Patience w;
                    while (load_acquire(&ra.flag[q]) < (unsigned long long)steps)
                        if (!w.more()) {
                            s_late = 1;
                            break;
                        }
                }
                __syncwarp();
                for (int k = warp; k < cnt_b; k += kRunNT / 32) {
                    const long long a = off_b + k;
                    if (MODE == NB_SUM_FIXED) {
                        Int128 t8[8];
#pragma unroll
                        for (int c = 0; c < 8; ++c) t8[c] = {0, 0};
                        for (int q = lane; q < ncta; q += 32) {
                            const longlong2 *pp =
                                reinterpret_cast<const longlong2 *>(ra.part) + (a * ncta + q) * 8;
                            longlong2 v[7];
#pragma unroll
                            for (int c = 0; c < 7; ++c) v[c] = __ldcg(&pp[c]);
#pragma unroll
                            for (int c = 0; c < 7; ++c) {
                                const unsigned long long l2 = t8[c].lo + (unsigned long long)v[c].y;
                                t8[c].hi += v[c].x + (l2 < t8[c].lo ? 1 : 0);
                                t8[c].lo = l2;
                            }
                        }
                        const Int128 t = warp_scatter8(t8, lane, AddI128());
                        const int e = lane >> 2;
                        if ((lane & 3) == 0 && e < kComp)
                            s_res[8 * k + e] = __dmul_rn(i128_to_double(t.hi, t.lo),
                                                         e < 3 ? Sc.inv[0] : (e < 6 ? Sc.inv[1] : Sc.inv[2]));
                    } else {
                        // per component: CTAs lane, lane + 32, ... in turn, then the fixed tree
                        double t8[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
                        for (int q = lane; q < ncta; q += 32) {
                            const double2 *pp = reinterpret_cast<const double2 *>(ra.part) + (a * ncta + q) * 4;
                            double2 v[4];
#pragma unroll
                            for (int c = 0; c < 4; ++c) v[c] = __ldcg(&pp[c]);
#pragma unroll
                            for (int c = 0; c < 4; ++c) {
                                t8[2 * c] += v[c].x;
                                if (c < 3) t8[2 * c + 1] += v[c].y;
                            }
                        }
                        const double t = warp_scatter8(t8, lane, AddF64());
                        const int e = lane >> 2;
                        if ((lane & 3) == 0 && e < kComp) s_res[8 * k + e] = t;
                    }
                }
            }
            __syncthreads();
            if (s_late) break;
            if (cnt_b <= kRunQuadMax) {
                // few particles: four lanes each
                if (warp * 8 < cnt_b) {
                    const int kq = tid >> 2, qd = tid & 3;
                    const bool active = kq < cnt_b;
                    const int kk = active ? kq : cnt_b - 1;
                    const int c = qd < 3 ? qd : 2;
                    const int li = s_blk[kk];
                    const bool ok = correct_particle_quad(L, li, per, tn_b, s_res[8 * kk + c],
                                                          s_res[8 * kk + 3 + c], ra.eta, ra.level_min,
                                                          ra.level_fixed, active);
                    if (active && qd == 0) {
                        if (!ok) {
                            atomicCAS(&ra.ctrl->err, 0, NB_ESTEP);
                            s_err = 1;
                        }
                        s_et[li] = tn_b + (1LL << (kTickBits - s_lev[li]));
                    }
                }
            } else if (tid < cnt_b) {
                const double *f = s_res + 8 * tid;
                const double ap[3] = {f[0], f[1], f[2]};
                const double kp[3] = {f[3], f[4], f[5]};
                const int li = s_blk[tid];
                if (!correct_particle(L, li, per, tn_b, ap, kp, ra.eta, ra.level_min, ra.level_fixed)) {
                    atomicCAS(&ra.ctrl->err, 0, NB_ESTEP);
                    s_err = 1;
                }
                s_et[li] = tn_b + (1LL << (kTickBits - s_lev[li]));
            }
            __syncthreads();
        }

        // 2. The first warp publishes the CTA's least end time with its count,
        // then reads everyone's: block time, stop decision, block size, offset.
        if (warp == 0) {
            long long mn = LLONG_MAX;
            for (int q = lane; q < m; q += 32) mn = min(mn, s_et[q]);
            mn = warp_min(mn);
            unsigned cnt = 0;
            for (int q = lane; q < m; q += 32) cnt += s_et[q] == mn;
            cnt = __reduce_add_sync(kFullR, cnt);
            ulonglong2 *const slot = ra.minrec + (epoch & 1u) * ncta;
            if (lane == 0)
                store128(&slot[r], {(unsigned long long)mn, (unsigned long long)(cnt | (s_err ? 0x80000000u : 0u)) |
                                                                ((unsigned long long)epoch << 32)});
            ulonglong2 rec[kRunPerLane];
#pragma unroll
            for (int u = 0; u < kRunPerLane; ++u)
                if (lane + 32 * u < ncta) rec[u] = load128(&slot[lane + 32 * u]);
            bool late = false;
#pragma unroll
            for (int u = 0; u < kRunPerLane; ++u)
                if (lane + 32 * u < ncta) {
                    Patience w;
                    while (tag_of(rec[u]) != epoch && !late) {
                        if (w.more()) rec[u] = load128(&slot[lane + 32 * u]);
                        else late = true;
                    }
                }
            long long tn = LLONG_MAX;
            unsigned err = 0;
#pragma unroll
            for (int u = 0; u < kRunPerLane; ++u)
                if (lane + 32 * u < ncta) {
                    tn = min(tn, (long long)rec[u].x);
                    err |= (unsigned)rec[u].y & 0x80000000u;
                }
            tn = warp_min(tn);
            unsigned na = 0, off = 0;
#pragma unroll
            for (int u = 0; u < kRunPerLane; ++u)
                if (lane + 32 * u < ncta && (long long)rec[u].x == tn) {
                    const unsigned c = (unsigned)rec[u].y & 0x7fffffffu;
                    na += c;
                    off += lane + 32 * u < r ? c : 0u;
                }
            na = __reduce_add_sync(kFullR, na);
            off = __reduce_add_sync(kFullR, off);
            err = __reduce_or_sync(kFullR, err);
            late = __any_sync(kFullR, late);
            if (lane == 0) {
                s_tn = tn;
                s_na = (int)na;
                s_off = (int)off;
                s_stop = err != 0 ? 1 : (tn > ra.t_end ? 2 : (steps >= ra.max_steps ? 1 : 0));
                if (late) s_late = 1;
            }
        }
        __syncthreads();
        if (s_late) break;
        const long long tn = s_tn;
        if (s_stop) {
            past_end = s_stop == 2;
            tn_end = tn;
            break;
        }
        const int na = s_na;
        // block members in ascending order: every warp counts the particles before its own
        int before = 0, cnt_own = 0;
        for (int g = 0; g * 32 < m; ++g) {
            const unsigned bal = __ballot_sync(kFullR, g * 32 + lane < m && s_et[g * 32 + lane] == tn);
            if (g < warp) before += __popc(bal);
            else if (g == warp) before += __popc(bal & ((1u << lane) - 1u));
            cnt_own += __popc(bal);
        }
        off_b = s_off;
        cnt_b = cnt_own;
        na_b = na;
        tn_b = tn;
        // Prediction, a warp to one axis of 32 particles: a warp has one FP64
        // instruction in flight, whatever its lanes.
        const bool member = tid < m && s_et[tid] == tn;
        if (member) s_blk[before] = tid;
        for (int task = warp; task < 3 * ((m + 31) / 32); task += kRunNT / 32) {
            const int c = task % 3, q = task / 3 * 32 + lane;
            if (q < m) {
                const double dt = ticks_to_time(tn - s_t[q]);
                const int e = c * per + q;
                double xp, vp;
                predict1hq(L.x[e], L.v[e], L.a[e], L.k[e], dt, half_dt(dt), div_core<3>(dt), xp, vp);
                float h, l, u;
                bool bad = false;
                split_ds_int(xp, h, l, bad);
                u = to_float_int(vp, bad);
                if (bad) split_rest(xp, vp, h, l, u);
                reinterpret_cast<float *>(&s_p[q])[c] = h;
                reinterpret_cast<float *>(&s_l[q])[c] = l;
                reinterpret_cast<float *>(&s_v[q])[c] = u;
            }
        }
        __syncthreads();
        unsigned mb = 0, vb = 0;
        if (member) {
            const float4 h = s_p[tid], l = s_l[tid], v = s_v[tid];
            float4 *const dst = ra.blk + 3 * (long long)(off_b + before);
            const unsigned long long tag = (unsigned long long)(epoch << kRunIndexBits | (unsigned)(i0 + tid)) << 32;
            auto put = [&](int q, float x, float y, float z) {
                store128(dst + q, {(unsigned long long)__float_as_uint(x) | (unsigned long long)__float_as_uint(y) << 32,
                                   (unsigned long long)__float_as_uint(z) | tag});
            };
            put(0, h.x, h.y, h.z);
            put(1, l.x, l.y, l.z);
            put(2, v.x, v.y, v.z);
        }
        if (MODE == NB_SUM_FIXED && tid < m) {
            const float4 v = s_v[tid];
            mb = __float_as_uint(fabsf(s_p[tid].w));   // a mass may be -0.0
            vb = __float_as_uint(__fadd_rn(__fadd_rn(fabsf(v.x), fabsf(v.y)), fabsf(v.z)));
        }
        if (MODE == NB_SUM_FIXED) {
            mb = __reduce_max_sync(kFullR, mb);
            vb = __reduce_max_sync(kFullR, vb);
            if (lane == 0) s_max[0][warp] = mb, s_max[1][warp] = vb;
            __syncthreads();
            // the bounds over all particles: published and read like the end times
            if (warp == 0) {
                mb = lane < kRunNT / 32 ? s_max[0][lane] : 0u;
                vb = lane < kRunNT / 32 ? s_max[1][lane] : 0u;
                mb = __reduce_max_sync(kFullR, mb);
                vb = __reduce_max_sync(kFullR, vb);
                ulonglong2 *const slot = ra.maxrec + (epoch & 1u) * ncta;
                if (lane == 0) store128(&slot[r], {(unsigned long long)mb, (unsigned long long)vb | ((unsigned long long)epoch << 32)});
                bool late = false;
                for (int q = lane; q < ncta; q += 32) {
                    Patience w;
                    ulonglong2 rec = load128(&slot[q]);
                    while (tag_of(rec) != epoch && !late) {
                        if (w.more()) rec = load128(&slot[q]);
                        else late = true;
                    }
                    mb = max(mb, (unsigned)rec.x);
                    vb = max(vb, (unsigned)rec.y);
                }
                mb = __reduce_max_sync(kFullR, mb);
                vb = __reduce_max_sync(kFullR, vb);
                late = __any_sync(kFullR, late);
                __syncwarp();
                if (lane == 0) {
                    s_max[0][0] = mb;
                    s_max[1][0] = vb;
                    if (late) s_late = 1;
                }
            }
            __syncthreads();
            if (s_late) break;
            const unsigned bounds[2] = {s_max[0][0], s_max[1][0]};
            scale_ok = fixed_scale(bounds, ra.eps2f, Sc);
            if (!scale_ok && tid == 0) {
                atomicCAS(&ra.ctrl->err, 0, kErrFixedScale);
                s_err = 1;   // the next stop decision ends the run
            }
        }

        // 3. force partials of every block particle over this CTA's particles
        bool ok = true;
        if (scale_ok) {
            int g = 1;
            while (g < 32 && g * 2 * na <= kRunNT) g <<= 1;
            switch (g) {
            case 1: ok = force_phase<MODE, 1>(ra, r, na, i0, m, epoch, s_p, s_l, s_v, Sc); break;
            case 2: ok = force_phase<MODE, 2>(ra, r, na, i0, m, epoch, s_p, s_l, s_v, Sc); break;
            case 4: ok = force_phase<MODE, 4>(ra, r, na, i0, m, epoch, s_p, s_l, s_v, Sc); break;
            case 8: ok = force_phase<MODE, 8>(ra, r, na, i0, m, epoch, s_p, s_l, s_v, Sc); break;
            case 16: ok = force_phase<MODE, 16>(ra, r, na, i0, m, epoch, s_p, s_l, s_v, Sc); break;
            default: ok = force_phase<MODE, 32>(ra, r, na, i0, m, epoch, s_p, s_l, s_v, Sc); break;
            }
        }
        if (!ok) s_late = 1;
        __syncthreads();
        if (s_late) break;
        ++steps;
        inter += (long long)na * (long long)(n - 1);
        if (tid == 0) store_release(&ra.flag[r], (unsigned long long)steps);
    }

    // the state, the last step's j records and block list, and the counters go back
    __syncthreads();
    if (s_late && tid == 0) atomicCAS(&ra.ctrl->err, 0, NB_ETIMEOUT);
    if (tid < m) {
        const int i = i0 + tid;
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            ra.s.x[(long long)c * n + i] = L.x[c * per + tid];
            ra.s.v[(long long)c * n + i] = L.v[c * per + tid];
            ra.s.a[(long long)c * n + i] = L.a[c * per + tid];
            ra.s.k[(long long)c * n + i] = L.k[c * per + tid];
        }
        ra.s.t[i] = s_t[tid];
        ra.s.lev[i] = s_lev[tid];
        if (steps > 0) {
            ra.j.pos_hi[i] = s_p[tid];
            ra.j.pos_lo[i] = s_l[tid];
            ra.j.vel[i] = s_v[tid];
        }
    }
    if (steps > 0 && tid < cnt_b) ra.act[off_b + tid] = i0 + s_blk[tid];
    if (r == 0 && tid == 0) {
        if (steps > 0) {
            ra.ctrl->t_next = tn_b;
            ra.ctrl->t_now = tn_b;
            ra.ctrl->n_active = na_b;
            ra.ctrl->steps += steps;
            ra.ctrl->interactions += inter;
        }
        if (past_end) {   // as the per-stage scheduler leaves it
            ra.ctrl->t_next = tn_end;
            ra.ctrl->n_active = 0;
        }
    }
}

}  // namespace

int run_layout(int n, int sms, int blocks_per_sm, int *ncta, int *per)
{
    // 32 particles per CTA up to 64 CTAs, then up to 64 particles per CTA
    // (64 CTAs at n = 4096), then one CTA per SM (measured on whole runs: more
    // CTAs share the force and the predictor but add to every exchange and to
    // the partials each block particle sums; above 4096 bodies the force
    // share wins)
    int p = (n + 63) / 64;
    if (p < 32) p = 32;
    if (p > 64) p = (n + sms - 1) / sms;
    if (p > kRunNT) return -1;
    const int c = (n + p - 1) / p;
    if (c > sms * blocks_per_sm || c > 32 * kRunPerLane) return -1;
    *ncta = c;
    *per = p;
    return 0;
}

int occupancy_run(int summation, int *blocks_per_sm)
{
    // at the largest particle count of a CTA, which any layout's CTA fits
    const int smem = kRunNT * kRunBytesPer;
    cudaError_t e;
    if (summation == NB_SUM_FIXED) {
        e = cudaFuncSetAttribute(k_run<NB_SUM_FIXED>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_run<NB_SUM_FIXED>, kRunNT, smem);
    } else {
        e = cudaFuncSetAttribute(k_run<NB_SUM_COMPENSATED>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_run<NB_SUM_COMPENSATED>, kRunNT, smem);
    }
    return e == cudaSuccess ? 0 : -1;
}

cudaError_t launch_check_wait(const unsigned long long *counter, long long limit_cycles, Ctrl *ctrl,
                              cudaStream_t st)
{
    k_check_wait<<<1, 1, 0, st>>>(counter, limit_cycles, ctrl);
    return cudaGetLastError();
}

cudaError_t launch_run(const RunArgs &ra, int summation, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.gridDim = dim3(ra.ncta);
    cfg.blockDim = dim3(kRunNT);
    cfg.dynamicSmemBytes = (size_t)ra.per * kRunBytesPer;
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (summation == NB_SUM_FIXED) return cudaLaunchKernelEx(&cfg, k_run<NB_SUM_FIXED>, ra);
    return cudaLaunchKernelEx(&cfg, k_run<NB_SUM_COMPENSATED>, ra);
}

}  // namespace nbk
