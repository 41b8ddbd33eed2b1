// k_sum.cu -- the force with the summation variants of Section 6.
//
// The paper contrasts GRAPE-6, which accumulates pair forces in 64-bit fixed
// point, with the GPU, which sums in single precision, and suggests sorting
// the forces and adding the smallest first.  These kernels evaluate the same
// single-precision pair terms on the double-single j records,
//
//   dx   = (xj_hi - xi_hi) + (xj_lo - xi_lo),   u = vj - vi        (per axis)
//   d2   = (dx0 dx0 + dx1 dx1) + dx2 dx2,        r2 = d2 + eps2
//   rv   = (dx0 u0 + dx1 u1) + dx2 u2
//   rinv = 1 / sqrt(r2),  rinv2 = rinv rinv,  mr = mj rinv,  mr3 = mr rinv2
//   b    = (-3 rv) rinv2
//   acc  = (mr3 Sa) dx,   jerk = (mr3 Sk) (u + b dx),   pot = -(mr Sp),
//
// every operation one IEEE single-precision operation rounded to nearest in
// that order (the __f*_rn intrinsics are never contracted into multiply-adds),
// so a CPU evaluating the same sequence gets the same bits.  The pair j = i
// and pairs with r2 = 0 contribute nothing.  Three summations:
//
//  NB_SUM_FIXED  Sa, Sk, Sp are powers of two chosen from bounds over all
//    particles so that every scaled term stays below 2^56; each term is
//    rounded to the nearest integer (ties to even) and the integers are summed
//    exactly in 128 bits.  Integer sums do not depend on their order, so the
//    result depends on neither the order of j, nor the j slices, nor which
//    CTA computes what.  (The rounding avoids float-to-int64 conversions, which
//    run on the FP64 pipe: three exact FP32 splits do it on the FP32 pipe.)
//  NB_SUM_FP32  per i an FP32 running sum over j = 0, 1, ... ; the terms are
//    evaluated in parallel, only the additions are in order.
//  NB_SUM_FP32_SORTED  one CTA per i: the pair-force magnitudes |mj dx/r^3|
//    as keys, a stable radix sort of (key, j), then the FP32 running sum in
//    increasing key (ties in increasing j).
#include <cfloat>
#include <type_traits>

#include "nb_device.cuh"

namespace nbk {
namespace {

using namespace dev;

constexpr unsigned kFull = 0xffffffffu;

// The largest single-precision mass and |vx| + |vy| + |vz| over all j, as
// float bits (non-negative floats order like their bits; the sign of a mass of
// -0.0 is cleared); bounds[] must be zero on entry.
__global__ void k_fixed_bounds(JDS J, int n, unsigned *bounds)
{
    unsigned mb = 0, vb = 0;
    for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n; j += gridDim.x * blockDim.x) {
        const float4 v = J.vel[j];
        const float v1 = __fadd_rn(__fadd_rn(fabsf(v.x), fabsf(v.y)), fabsf(v.z));
        mb = max(mb, __float_as_uint(fabsf(J.pos_hi[j].w)));
        vb = max(vb, __float_as_uint(v1));
    }
    mb = __reduce_max_sync(kFull, mb);
    vb = __reduce_max_sync(kFull, vb);
    if ((threadIdx.x & 31) == 0) {
        atomicMax(&bounds[0], mb);
        atomicMax(&bounds[1], vb);
    }
}

// Two pairs (j, j + 1) into the tile's split sums; the pair j = i adds zeros,
// so every tile adds all its terms.
template <bool GUARD>
__device__ __forceinline__ void pair_fixed2(const Side2 &Js, const Side2 &N, float eps2, const Scale &S,
                                            unsigned a[3][7], int j = 0, int i = 1)
{
    float2 t[7];
    pair_rn2<false>(Js, N, eps2, S.sc[0], S.sc[1], S.sc[2], t);
#pragma unroll
    for (int q = 0; q < 7; ++q) {
        if (GUARD) t[q] = make_float2(j == i ? 0.0f : t[q].x, j + 1 == i ? 0.0f : t[q].y);
        split_add2(t[q], a[0][q], a[1][q], a[2][q]);
    }
}

// i-parallel like the DS kernel: a CTA owns NT active i, one per thread, and
// one j slice, tiles of TL j in shared memory; 64-bit tile sums, 128-bit
// totals; with several slices the totals go to the partial buffer as (hi, lo)
// pairs.  The j side lies in shared memory component by component, so that
// one 16-byte read gives a component of four j, two packed operands: every
// single-precision operation of the terms and of their splitting then serves
// two pairs.  Bound by the FMA pipe (about 103 operations a pair, of which 49
// split the terms); the scalar form was bound by issue at 132 instructions a
// pair.  65536 bodies all active: 17.4 ms -> 14.6 ms packed, 13.5 ms with one
// CTA per work item (grid_summed), 13.2 ms with more slices and ten CTAs a SM.
template <int NT>
__global__ void __launch_bounds__(NT, kFixCtas) k_force_fixed(ForceArgs fa, JDS J, SumArgs sa)
{
    const ForcePlan F = load_plan(fa);
    const int na = F.na;
    if (na <= 0) return;
    const float eps2 = (float)fa.eps2;
    Scale S;
    if (!fixed_scale(sa.bounds, eps2, S)) {
        if (blockIdx.x == 0 && threadIdx.x == 0) atomicCAS(fa.err, 0, kErrFixedScale);
        return;
    }
    const Plan P = F.p;
    long long *part = reinterpret_cast<long long *>(fa.part);
    constexpr int TL = 2 * NT;   // j per shared-memory tile; TL 2^22 stays below 2^31 (split_add)
    __shared__ float4 s_j[10][TL / 4];
    float *const sj = reinterpret_cast<float *>(s_j);
    const int tid = threadIdx.x;

    for (int w = blockIdx.x; w < P.items; w += gridDim.x) {
        const int ib = w % P.n_iblk;
        const int sl = w / P.n_iblk;
        const int j0 = sl * P.jslice;
        const int j1 = min(fa.n, j0 + P.jslice);

        const int a = ib * NT + tid;
        const int ia = a < na ? a : -1;
        const int ii = clamp_index(fa.act[a < na ? a : 0], fa.n);
        const Side2 N = side2_neg(J.pos_hi[ii], J.pos_lo[ii], J.vel[ii]);
        long long hi[7];
        unsigned long long lo[7];
#pragma unroll
        for (int q = 0; q < 7; ++q) hi[q] = 0, lo[q] = 0;

        for (int jt = j0; jt < j1; jt += TL) {
            __syncthreads();
#pragma unroll
            for (int u = 0; u < TL / NT; ++u) {
                const int t = tid + u * NT, j = jt + t;
                const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);  // mass 0: contributes 0
                const float4 p = j < j1 ? J.pos_hi[j] : z, l = j < j1 ? J.pos_lo[j] : z,
                             v = j < j1 ? J.vel[j] : z;
                const float c[10] = {p.x, p.y, p.z, l.x, l.y, l.z, v.x, v.y, v.z, p.w};
#pragma unroll
                for (int e = 0; e < 10; ++e) sj[e * TL + t] = c[e];
            }
            __syncthreads();
            const int jc = (min(TL, j1 - jt) + 3) & ~3;   // whole reads of four; the padding adds zeros
            unsigned ch[3][7];
#pragma unroll
            for (int q = 0; q < 7; ++q) ch[0][q] = ch[1][q] = ch[2][q] = 0u;
            auto four = [&](int jj, auto guard) {
                float4 c[10];
#pragma unroll
                for (int e = 0; e < 10; ++e) c[e] = s_j[e][jj / 4];
#pragma unroll
                for (int h = 0; h < 2; ++h) {
                    Side2 Js;
#pragma unroll
                    for (int e = 0; e < 3; ++e) {
                        Js.h[e] = h ? make_float2(c[e].z, c[e].w) : make_float2(c[e].x, c[e].y);
                        Js.l[e] = h ? make_float2(c[3 + e].z, c[3 + e].w) : make_float2(c[3 + e].x, c[3 + e].y);
                        Js.v[e] = h ? make_float2(c[6 + e].z, c[6 + e].w) : make_float2(c[6 + e].x, c[6 + e].y);
                    }
                    Js.m = h ? make_float2(c[9].z, c[9].w) : make_float2(c[9].x, c[9].y);
                    pair_fixed2<decltype(guard)::value>(Js, N, eps2, S, ch, jt + jj + 2 * h, ii);
                }
            };
            if (__any_sync(kFull, (unsigned)(ii - jt) < (unsigned)TL)) {
                for (int jj = 0; jj < jc; jj += 4) four(jj, std::true_type());
            } else {
                for (int jj = 0; jj < jc; jj += 4) four(jj, std::false_type());
            }
#pragma unroll
            for (int q = 0; q < 7; ++q)
                add128(hi[q], lo[q], tile_sum(ch[0][q], ch[1][q], ch[2][q], (unsigned)jc));
        }

        if (ia < 0) continue;
        if (P.S == 1) {
            double res[kComp];
#pragma unroll
            for (int q = 0; q < 7; ++q)
                res[q] = __dmul_rn(i128_to_double(hi[q], lo[q]), S.inv[q < 3 ? 0 : (q < 6 ? 1 : 2)]);
            store_result(fa.out, ia, res);
        } else {
#pragma unroll
            for (int q = 0; q < 7; ++q) {
                long long *pp = part + 2 * (((long long)sl * kComp + q) * na + ia);
                pp[0] = hi[q];
                pp[1] = (long long)lo[q];
            }
        }
    }
}

// Sum of the slices' 128-bit totals (exact, any order) and conversion.
__global__ void k_fixed_combine(ForceArgs fa, SumArgs sa)
{
    const ForcePlan F = load_plan(fa);
    const int na = F.na;
    if (na <= 0) return;
    const Plan P = F.p;
    if (P.S == 1) return;
    Scale S;
    if (!fixed_scale(sa.bounds, (float)fa.eps2, S)) return;
    const long long *part = reinterpret_cast<const long long *>(fa.part);
    const long long total = (long long)na * kComp;
    for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
         e += (long long)gridDim.x * blockDim.x) {
        const int c = (int)(e / na), a = (int)(e % na);
        long long hi = 0;
        unsigned long long lo = 0;
        for (int q = 0; q < P.S; ++q) {
            const long long *pp = part + 2 * (((long long)q * kComp + c) * na + a);
            const unsigned long long l2 = lo + (unsigned long long)pp[1];
            hi += pp[0] + (l2 < lo ? 1 : 0);
            lo = l2;
        }
        const double inv = c < 3 ? S.inv[0] : (c < 6 ? S.inv[1] : S.inv[2]);
        write_combined(fa.out, c, a, __dmul_rn(i128_to_double(hi, lo), inv));
    }
}

// Adds 4 N4 values of s to run in order.  Four reads are in flight while the
// sixteen values before them are added (64 clocks, a read takes about 30);
// left to the compiler the reads end up just ahead of their additions, 10
// clocks a value instead of 4.  The reads are volatile to stay where they are.
__device__ __forceinline__ float4 read_early(const float4 *p)
{
    float4 v;
    const unsigned a = (unsigned)__cvta_generic_to_shared(p);
    asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(a));
    return v;
}
__device__ __forceinline__ float add4(float run, const float4 &t)
{
    return __fadd_rn(__fadd_rn(__fadd_rn(__fadd_rn(run, t.x), t.y), t.z), t.w);
}
template <int N4>
__device__ __forceinline__ float add_in_order(const float4 *s, float run)
{
    static_assert(N4 % 4 == 0, "whole groups of reads");
    float4 a[4];
#pragma unroll
    for (int u = 0; u < 4; ++u) a[u] = read_early(s + u);
#pragma unroll 2
    for (int q = 4; q < N4; q += 4) {
        float4 b[4];
#pragma unroll
        for (int u = 0; u < 4; ++u) b[u] = read_early(s + q + u);
#pragma unroll
        for (int u = 0; u < 4; ++u) run = add4(run, a[u]), a[u] = b[u];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) run = add4(run, a[u]);
    return run;
}

// ---------------------------------------------------------------------------
// FP32 running sum in index order.  The order fixes one chain of additions per
// output (4 cycles a term), but nothing fixes who evaluates the terms: a CTA
// owns I active particles; 16 warps evaluate the seven terms of a tile of T
// sources, lane per source, into shared memory while 4 warps (one per
// scheduler) add the tile before it in index order, one lane per (particle,
// component).  Two tiles alternate with one barrier a tile.  A pair left out
// (j = i, r2 = 0) and the padding past n enter as -0, which changes no sum.
//
// Bounds: with many particles the term evaluation's issue slots (two
// particles share every packed operation), with few the chain of additions.
// I spreads the block evenly over the resident CTAs, one per SM; T grows as I
// shrinks (the buffers keep their size) so that the barrier stays a small part
// of the tile's chain.  1820 active on 65536 bodies: 458 us; one thread per i
// evaluating and adding its own terms kept 15 SMs busy and took 9.54 ms.  Of
// the steps between, all with the same bits: tiles of 128 sources 627 us,
// larger tiles and the next records loaded ahead 583 us, packed pairs and the
// short 1/sqrt 502 us, tile lengths as compile-time constants 458 us.

constexpr int kSeqI = 15;             // active particles per CTA at most
constexpr int kSeqTermWarps = 16;     // warps that evaluate terms
constexpr int kSeqSumWarps = kSeqNT / 32 - kSeqTermWarps;
static_assert(kSeqSumWarps * 32 >= kSeqI * kComp, "one summing lane per (particle, component)");

// Particles per CTA and sources per tile for a block of na on `slots` CTAs:
// the fewest rounds of at most kSeqI particles, split evenly.
__host__ __device__ inline void seq_shape(int na, int slots, int &I, int &T)
{
    const int rounds = cdiv(na, (long long)slots * kSeqI);
    I = cdiv(na, (long long)slots * rounds);
    T = I > 7 ? 256 : (I > 3 ? 512 : 1024);
}

// Rows of T terms are T + 4 floats apart: the summing lanes' 16-byte reads of
// eight rows then fall into different banks.
__host__ __device__ constexpr int seq_row(int T) { return T + 4; }
constexpr int kSeqBufFloats = kSeqI * kComp * seq_row(256);   // the largest of the shapes
static_assert(7 * seq_row(512) <= kSeqI * seq_row(256) && 3 * seq_row(1024) <= kSeqI * seq_row(256),
              "every shape fits the buffers");
constexpr int kSeqSmem = 2 * kSeqBufFloats * (int)sizeof(float);

template <int T>
__device__ __forceinline__ void seq_groups(const ForceArgs &fa, const JDS &J, int na, int I)
{
    extern __shared__ float4 s_dyn[];
    float *const buf = reinterpret_cast<float *>(s_dyn);
    __shared__ float2 s_i[(kSeqI + 1) / 2][10];   // two particles' records, negated, component by component
    __shared__ int s_ii[kSeqI + 1];
    __shared__ float s_sum[kSeqI * kComp];
    constexpr int row = seq_row(T), nsub = T / 32;
    const float eps2 = (float)fa.eps2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, n = fa.n;
    const int ntile = cdiv(n, T), ngrp = cdiv(na, I);
    // term warp w takes sub-tiles w mod nsub, + 16, ... and, with fewer
    // sub-tiles than warps, every qstep-th pair of particles
    const int qstep = nsub < kSeqTermWarps ? kSeqTermWarps / nsub : 1;
    const int sub0 = nsub < kSeqTermWarps ? warp % nsub : warp, q0 = nsub < kSeqTermWarps ? warp / nsub : 0;
    const int jlane = sub0 * 32 + lane;   // this lane's first source within a tile
    for (int grp = blockIdx.x; grp < ngrp; grp += gridDim.x) {
        const int a0 = grp * I, cnt = min(I, na - a0), npair = (cnt + 1) / 2;
        __syncthreads();
        if (tid < 2 * npair) {   // an odd count repeats the last particle, unstored
            const int i = clamp_index(fa.act[a0 + min(tid, cnt - 1)], n);
            const float4 p = J.pos_hi[i], l = J.pos_lo[i], v = J.vel[i];
            const float c[9] = {p.x, p.y, p.z, l.x, l.y, l.z, v.x, v.y, v.z};
            float *const d = reinterpret_cast<float *>(s_i[tid >> 1]) + (tid & 1);
#pragma unroll
            for (int e = 0; e < 9; ++e) d[2 * e] = -c[e];
            s_ii[tid] = i;
        }
        __syncthreads();
        const int chain = tid - kSeqTermWarps * 32;   // summing lanes: particle * 7 + component
        float sum = 0.0f;
        // a term warp's next source records are loaded while it works on the
        // present ones (the index of padding lanes is clamped)
        float4 np, nl, nv;
        if (warp < kSeqTermWarps) {
            const int jc = min(jlane, n - 1);
            np = J.pos_hi[jc], nl = J.pos_lo[jc], nv = J.vel[jc];
        }
        for (int k = 0; k <= ntile; ++k) {
            if (warp < kSeqTermWarps) {
                if (k < ntile) {
                    float *const dst = buf + (k & 1) * kSeqBufFloats;
                    for (int sub = sub0; sub < nsub; sub += kSeqTermWarps) {
                        const int jj = sub * 32 + lane, j = k * T + jj;
                        const Side2 Js = side2(np, nl, nv, np, nl, nv);
                        const int jn = min(sub + kSeqTermWarps < nsub ? j + kSeqTermWarps * 32
                                                                      : (k + 1) * T + jlane, n - 1);
                        np = J.pos_hi[jn], nl = J.pos_lo[jn], nv = J.vel[jn];
                        const int j0 = j - lane;
                        const bool edge = j0 + 32 > n || !(eps2 > 0.0f);
                        for (int q = q0; q < npair; q += qstep) {
                            Side2 N;
#pragma unroll
                            for (int c = 0; c < 3; ++c)
                                N.h[c] = s_i[q][c], N.l[c] = s_i[q][3 + c], N.v[c] = s_i[q][6 + c];
                            float2 t[7];
                            const float2 r2 = pair_rn2<true>(Js, N, eps2, 1.0f, 1.0f, 1.0f, t);
                            const int ia = s_ii[2 * q], ib = s_ii[2 * q + 1];
                            // pairs to leave out can only be here (uniform in the warp)
                            if ((unsigned)(ia - j0) < 32u || (unsigned)(ib - j0) < 32u || edge) {
                                const bool oa = j < n && j != ia && r2.x != 0.0f;
                                const bool ob = j < n && j != ib && r2.y != 0.0f;
#pragma unroll
                                for (int c = 0; c < 7; ++c)
                                    t[c] = make_float2(oa ? t[c].x : -0.0f, ob ? t[c].y : -0.0f);
                            }
                            float *const d = dst + 2 * q * kComp * row + jj;
#pragma unroll
                            for (int c = 0; c < 7; ++c) d[c * row] = t[c].x;
                            if (2 * q + 1 < cnt)
#pragma unroll
                                for (int c = 0; c < 7; ++c) d[(kComp + c) * row] = t[c].y;
                        }
                    }
                }
            } else if (k > 0 && chain < cnt * kComp) {
                sum = add_in_order<T / 4>(reinterpret_cast<const float4 *>(buf + ((k - 1) & 1) * kSeqBufFloats +
                                                                           chain * row), sum);
            }
            __syncthreads();
        }
        if (chain >= 0 && chain < cnt * kComp) s_sum[chain] = sum;
        __syncthreads();
        if (tid < cnt) {
            double res[kComp];
#pragma unroll
            for (int c = 0; c < kComp; ++c) res[c] = (double)s_sum[tid * kComp + c];
            store_result(fa.out, a0 + tid, res);
        }
    }
}

__global__ void __launch_bounds__(kSeqNT, 1) k_force_seq(ForceArgs fa, JDS J, int slots)
{
    const int na = read_na(fa);
    if (na <= 0) return;
    int I, T;
    seq_shape(na, slots, I, T);
    if (T == 256) seq_groups<256>(fa, J, na, I);
    else if (T == 512) seq_groups<512>(fa, J, na, I);
    else seq_groups<1024>(fa, J, na, I);
}

// ---------------------------------------------------------------------------
// FP32 running sum, smallest pair force first: one CTA per active i.  The keys
// |mj dx/r^3| are sorted stably by j and the terms added in that order.
//  1. a histogram of the keys over bins of 1/32 octave, and where a bin holds
//     more than 2048 items (a particle far out sees all others at one distance)
//     a second one of finer bins over the keys' own range: with bins of at most
//     2048 a chunk stays within the 4096 items that shared memory takes;
//  2. consecutive bins make chunks of up to 4096 items (about 2048 each); the
//     items (key bits << 32 | j) go to their chunk in the CTA's scratch, keys
//     evaluated again rather than stored and read: 8 bytes written and read
//     per item in all;
//  3. chunk by chunk, in increasing key: a bucket sort of (key, j) in shared
//     memory, then the terms.
// While seven warps evaluate a tile's terms, seven lanes of the eighth add the
// tile before it in order, one component each (4 clocks an item), so four CTAs
// share an SM, each in its own phase.
//
// Where a bin still holds more than 2048 items (many equal keys) or there are
// more than 255 chunks, all items are sorted in the scratch instead, by a stable
// LSD radix sort with a pass per key byte (a byte that all keys share is left
// out).  An item's rank within a pass is that among the equal digits of its
// warp (match_any and the warp's running counts in shared memory) plus the
// counts of the earlier warps and tiles; stability keeps equal keys in index
// order.  Its scattered stores to a footprint beyond the L2 are what that waits
// for.  Up to kChunks kChunk particles, where it is the exception, it moves
// indices alone and evaluates their keys again in every pass, so that a CTA's
// scratch is n words (sort_scratch_size); above, keyed items in two arrays.
//
// 1820 active on 65536 bodies: 5.1 ms (5.4 with the scratch sort in place of the
// finer bins, by keyed items, and 6.8 by indices; a radix sort of the chunks 6.1,
// the scratch sort alone 6.6); one CTA of 1024 threads per SM, ranking one item a
// thread between five barriers and adding after evaluating, 18.6 ms.

constexpr int kSortW = kSortNT / 32;
constexpr int kSortK = 16;                        // items per thread of a chunk or tile
constexpr int kSortTile = kSortNT * kSortK;
constexpr int kBinBits = 13, kBins = 1 << kBinBits;   // bins of the key's upper bits
constexpr int kBinShift = 18;
static_assert((0x7f7fffff >> kBinShift) < kBins && 2 * kChunk <= kSortTile, "keys have a bin, chunks fit");
constexpr int kSortSum = (kSortW - 1) * 32;       // items per tile of the sum: one per term lane
constexpr int kSortRow = kSortSum + 4;

struct SortShared {
    union {
        unsigned hist[kBins];                    // 1: histogram; the scratch sort's [4][256]
        unsigned long long item[kSortTile];      // 3: the chunk
    } a;
    unsigned char id[kBins];                     // chunk of a bin
    union {
        unsigned off[kSortW][256];               // counts, then offsets, of a warp's digits
        unsigned bucket[2048];                   // chunk: items per bucket, then places
        float4 t[2][7][kSortRow / 4];            // two tiles of terms
    } u;
    unsigned start[kChunks + 2];                 // first item of a chunk
    unsigned next[kChunks + 1];                  // place of its next item
    unsigned base[256];
    unsigned scan[kSortW], lo[kSortW], hi[kSortW];
    int cnt;
};

// (Functions that are not inlined take it from here, to know that it is shared memory.)
__device__ __forceinline__ SortShared &sort_shared()
{
    extern __shared__ float4 s_sorted[];
    return *reinterpret_cast<SortShared *>(s_sorted);
}

// Exclusive sum over the CTA's threads (a barrier before and after use of s).
__device__ __forceinline__ unsigned cta_exclusive(unsigned v, unsigned *s, int lane, int warp)
{
    unsigned incl = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const unsigned y = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += y;
    }
    if (lane == 31) s[warp] = incl;
    __syncthreads();
    unsigned before = incl - v;
    for (int w = 0; w < warp; ++w) before += s[w];
    return before;
}

// Ranks of a warp's K rows of 32 items (digit(k), or -1: none) among the equal
// digits of its rows so far, two 16-bit ranks a register; cnt[256] ends with
// the warp's counts.
template <int K, typename Digit>
__device__ __forceinline__ void warp_ranks(Digit digit, unsigned (&rank)[K / 2], unsigned *cnt, int lane, int rows)
{
    const unsigned lt = (1u << lane) - 1u;
#pragma unroll
    for (int q = 0; q < 256 / 32; ++q) cnt[q * 32 + lane] = 0;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < K; ++k) {
        if (k % 2 == 0) rank[k / 2] = 0;
        if (k < rows) {
            const int d = digit(k);
            const unsigned peers = __match_any_sync(kFull, d);
            const unsigned old = d >= 0 ? cnt[d] : 0u;
            rank[k / 2] |= (old + __popc(peers & lt)) << (16 * (k % 2));
            __syncwarp();
            if (d >= 0 && (peers & lt) == 0) cnt[d] = old + __popc(peers);
            __syncwarp();
        }
    }
}
template <int H>
__device__ __forceinline__ unsigned rank_of(const unsigned (&rank)[H], int k)
{
    return (rank[k / 2] >> (16 * (k % 2))) & 0xffffu;
}

// Two j's keys, ~0 for a pair that is left out.  The sign is cleared: a mass of
// -0.0 has the key -0.0, whose bits lie past the last bin (its terms are zeros,
// which change no running sum wherever they stand).
__device__ __forceinline__ uint2 sort_keys(const JDS &J, int j0, int j1, int n, int i, const Side2 &N, float eps2)
{
    const int c0 = min(j0, n - 1), c1 = min(j1, n - 1);
    const Side2 Js = side2(J.pos_hi[c0], J.pos_lo[c0], J.vel[c0], J.pos_hi[c1], J.pos_lo[c1], J.vel[c1]);
    float2 r2;
    const float2 key = pair_key2(Js, N, eps2, r2);
    return make_uint2(j0 < n && j0 != i && r2.x != 0.0f ? __float_as_uint(fabsf(key.x)) : ~0u,
                      j1 < n && j1 != i && r2.y != 0.0f ? __float_as_uint(fabsf(key.y)) : ~0u);
}

// Adds the terms of sorted items 0 .. total - 1 (index by `at`) to run, which
// lane c of warp 0 holds for component c.
template <typename At>
__device__ __forceinline__ void sum_sorted(SortShared &sh, const JDS &J, int i, float eps2, int total, At at, float &run)
{
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    float xh[3], xl[3], vi[3];
    load_i(J, i, xh, xl, vi);
    const int ntile = cdiv(total, kSortSum), q0 = (warp - 1) * 32 + lane;
    // a lane's next source record is loaded while it works on the present one
    float4 p, l, v;
    if (warp > 0 && ntile > 0) {
        const int j = at(min(q0, total - 1));
        p = J.pos_hi[j], l = J.pos_lo[j], v = J.vel[j];
    }
    for (int k = 0; k <= ntile; ++k) {
        if (warp > 0) {
            if (k < ntile) {
                const int e = k * kSortSum + q0;
                const int j = at(min(e + kSortSum, total - 1));
                const float4 np = J.pos_hi[j], nl = J.pos_lo[j], nv = J.vel[j];
                float t[7];
                pair_rn(p, l, v, xh, xl, vi, eps2, 1.0f, 1.0f, 1.0f, t);
                p = np, l = nl, v = nv;
                float *const d = reinterpret_cast<float *>(sh.u.t[k & 1]) + q0;
#pragma unroll
                for (int c = 0; c < 7; ++c) d[c * kSortRow] = e < total ? t[c] : -0.0f;   // -0 changes no sum
            }
        } else if (k > 0 && lane < 7) {
            run = add_in_order<kSortSum / 4>(sh.u.t[(k - 1) & 1][lane], run);
        }
        __syncthreads();
    }
}

// An item of the scratch sort: key and index where the scratch has room for two
// arrays of them; else the index alone, its key evaluated again for every pass.
template <typename Item>
struct SortItem {
    static constexpr bool kKeyed = sizeof(Item) == 8;
    static __device__ __forceinline__ Item make(unsigned key, int j)
    {
        return kKeyed ? (Item)((unsigned long long)key << 32 | (unsigned)j) : (Item)j;
    }
};

// The scratch sort: all n items by four passes between A and B; the sorted array,
// and in sh.cnt how many of its items are pairs to add.
template <typename Item>
__device__ __forceinline__ const Item *sort_scratch(SortShared &sh, const JDS &J, int i, int n, float eps2, Item *A,
                                                 Item *B)
{
    constexpr int NT = kSortNT;
    using It = SortItem<Item>;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Side2 N = side2_neg(J.pos_hi[i], J.pos_lo[i], J.vel[i]);
    unsigned(*hist)[256] = reinterpret_cast<unsigned(*)[256]>(sh.a.hist);
#pragma unroll
    for (int q = 0; q < 4; ++q) hist[q][tid] = 0;
    if (tid == 0) sh.cnt = 0;
    __syncthreads();
    int cnt = 0;
    for (int j = tid; j < n; j += 2 * NT) {
        const uint2 key = sort_keys(J, j, j + NT, n, i, N, eps2);
        cnt += (key.x != ~0u) + (key.y != ~0u);
        A[j] = It::make(key.x, j);
#pragma unroll
        for (int q = 0; q < 4; ++q) atomicAdd(&hist[q][(key.x >> (8 * q)) & 255u], 1u);
        if (j + NT < n) {
            A[j + NT] = It::make(key.y, j + NT);
#pragma unroll
            for (int q = 0; q < 4; ++q) atomicAdd(&hist[q][(key.y >> (8 * q)) & 255u], 1u);
        }
    }
    cnt = __reduce_add_sync(kFull, cnt);
    if (lane == 0) atomicAdd(&sh.cnt, cnt);
    __syncthreads();
    Item *src = A, *dst = B;
    for (int pass = 0; pass < 4; ++pass) {
        const unsigned mine = hist[pass][tid];
        if (__syncthreads_or(mine == (unsigned)n)) continue;   // one digit for all
        sh.base[tid] = cta_exclusive(mine, sh.scan, lane, warp);   // kept by this thread only
        for (int t0 = 0; t0 < n; t0 += kSortTile) {
            Item item[kSortK];
            unsigned rank[kSortK / 2], dig[kSortK / 4];   // dig: four digits a register
            const int w0 = t0 + warp * (kSortK * 32) + lane;
#pragma unroll
            for (int k = 0; k < kSortK; ++k) item[k] = w0 + k * 32 < n ? src[w0 + k * 32] : (Item)0;
            if (!It::kKeyed) {
#pragma unroll
                for (int k = 0; k < kSortK; k += 2) {
                    const uint2 key = sort_keys(J, (int)item[k], (int)item[k + 1], n, i, N, eps2);
                    const unsigned two = ((key.x >> (8 * pass)) & 255u) | ((key.y >> (8 * pass)) & 255u) << 8;
                    dig[k / 4] = k % 4 == 0 ? two : dig[k / 4] | two << 16;
                }
            }
            auto digit = [&](int k) {
                const unsigned d = It::kKeyed ? (unsigned)((unsigned long long)item[k] >> (32 + 8 * pass))
                                              : dig[k / 4] >> (8 * (k % 4));
                return w0 + k * 32 < n ? (int)(d & 255u) : -1;
            };
            warp_ranks<kSortK>(digit, rank, sh.u.off[warp], lane, kSortK);
            __syncthreads();
            unsigned run = sh.base[tid];
#pragma unroll
            for (int w = 0; w < kSortW; ++w) {
                const unsigned c = sh.u.off[w][tid];
                sh.u.off[w][tid] = run;
                run += c;
            }
            sh.base[tid] = run;
            __syncthreads();
#pragma unroll
            for (int k = 0; k < kSortK; ++k)
                if (w0 + k * 32 < n) dst[sh.u.off[warp][digit(k)] + rank_of(rank, k)] = item[k];
            __syncwarp();   // the warp's offsets are cleared next
        }
        __syncthreads();
        Item *tmp = src;
        src = dst;
        dst = tmp;
    }
    return src;
}

// All terms of particle i by the scratch sort.
template <typename Item>
__device__ __noinline__ float sum_in_scratch(const JDS J, int i, int n, float eps2, Item *A)
{
    SortShared &sh = sort_shared();
    const Item *sorted = sort_scratch(sh, J, i, n, eps2, A, A + n);
    float run = 0.0f;
    sum_sorted(sh, J, i, eps2, sh.cnt, [&](int q) { return (int)(unsigned)sorted[q]; }, run);
    return run;
}

// Chunk of cnt <= kSortTile items from src sorted into sh.a.item, by buckets:
// the chunk's key range over 2048 buckets, a place in its bucket for every
// item in any order (an atomic counter), then its rank among the bucket's items,
// which are compared as (key, j).  A bucket holds one or two items where the
// keys are spread; many equal keys cost their square, so a chunk with more than
// kCrowd items in a bucket is sorted by sort_crowded instead.
constexpr int kBuckets = 2048;
constexpr unsigned kCrowd = 128;

// The chunk's items, in any order in sh.a.item, sorted by a bitonic network whose
// merges begin with mirrored partners, so that all comparisons point upwards and
// those past the end can be left out.  Thread t has the pairs t, t + NT, ... of a
// stage: in spans of 64 items or less a warp stays within 64 items of its own.
// 152 active of 65536 bodies in 64 points: 1.10 ms, 5.18 with the buckets ranked
// by comparisons, 1.21 with the sort of all items by one CTA of 1024 threads an SM;
// in 256 points 1.14, 1.83, 1.22; on a lattice 1.30, 2.03, 1.40.  One pair at a
// time instead of four took 1.39, 1.45 and 1.59 (the pairs' reads are waited for).
__device__ __forceinline__ void sort_crowded(SortShared &sh, int cnt)
{
    constexpr int U = 4;   // pairs on their way at once
    __syncthreads();
    for (int k = 2; k < 2 * cnt; k <<= 1)
        for (int d = k >> 1; d > 0; d >>= 1) {
            const int mirror = d == k >> 1 ? -1 : 0;
            auto lower = [&](int t) { return 2 * t - (t & (d - 1)); };
            for (int t = threadIdx.x; lower(t) < cnt; t += U * kSortNT) {
                unsigned long long x[U], y[U];
                int a[U], b[U];
#pragma unroll
                for (int u = 0; u < U; ++u) {
                    const int o = (t + u * kSortNT) & (d - 1);
                    a[u] = lower(t + u * kSortNT);
                    b[u] = a[u] + d + ((d - 1 - 2 * o) & mirror);
                    x[u] = y[u] = 0;
                    if (b[u] < cnt) x[u] = sh.a.item[a[u]], y[u] = sh.a.item[b[u]];
                }
#pragma unroll
                for (int u = 0; u < U; ++u)
                    if (x[u] > y[u]) sh.a.item[a[u]] = y[u], sh.a.item[b[u]] = x[u];
            }
            if (d > 32 || (d == 1 && k >= 64)) __syncthreads();
            else __syncwarp();
        }
}

__device__ __forceinline__ void sort_chunk(SortShared &sh, const unsigned long long *src, int cnt)
{
    constexpr int NT = kSortNT, kOwn = kBuckets / NT;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    unsigned long long v[kSortK];
    unsigned lo = ~0u, hi = 0u;
#pragma unroll
    for (int k = 0; k < kSortK; ++k) {
        const int q = k * NT + tid;
        v[k] = q < cnt ? src[q] : ~0ULL;
        if (q < cnt) {
            lo = min(lo, (unsigned)(v[k] >> 32));
            hi = max(hi, (unsigned)(v[k] >> 32));
        }
    }
#pragma unroll
    for (int q = 0; q < kOwn; ++q) sh.u.bucket[q * NT + tid] = 0;
    lo = __reduce_min_sync(kFull, lo);
    hi = __reduce_max_sync(kFull, hi);
    if (lane == 0) sh.lo[warp] = lo, sh.hi[warp] = hi;
    __syncthreads();
#pragma unroll
    for (int w = 0; w < kSortW; ++w) lo = min(lo, sh.lo[w]), hi = max(hi, sh.hi[w]);
    const int shift = max(0, 21 - __clz(hi - lo));   // (hi - lo) >> shift < 2048
    auto bucket = [&](unsigned long long x) { return ((unsigned)(x >> 32) - lo) >> shift; };
#pragma unroll
    for (int k = 0; k < kSortK; ++k)
        if (k * NT + tid < cnt) atomicAdd(&sh.u.bucket[bucket(v[k])], 1u);
    __syncthreads();
    unsigned c[kOwn], sum = 0;
#pragma unroll
    for (int q = 0; q < kOwn; ++q) c[q] = sh.u.bucket[tid * kOwn + q], sum += c[q];
    unsigned at = cta_exclusive(sum, sh.scan, lane, warp), most = 0;
#pragma unroll
    for (int q = 0; q < kOwn; ++q) {
        sh.u.bucket[tid * kOwn + q] = at;
        at += c[q];
        most = max(most, c[q]);
    }
    if (__syncthreads_or(most > kCrowd)) {
#pragma unroll
        for (int k = 0; k < kSortK; ++k)
            if (k * NT + tid < cnt) sh.a.item[k * NT + tid] = v[k];
        sort_crowded(sh, cnt);
        return;
    }
#pragma unroll
    for (int k = 0; k < kSortK; ++k)
        if (k * NT + tid < cnt) sh.a.item[atomicAdd(&sh.u.bucket[bucket(v[k])], 1u)] = v[k];
    __syncthreads();
    // a bucket's counter now stands at its end, the start of the next
    unsigned place[kSortK / 2];
#pragma unroll
    for (int k = 0; k < kSortK; ++k) {
        if (k % 2 == 0) place[k / 2] = 0;
        if (k * NT + tid < cnt) {
            const unsigned d = bucket(v[k]), e = sh.u.bucket[d];
            unsigned q = d ? sh.u.bucket[d - 1] : 0u, r = q;
            for (; q < e; ++q) r += sh.a.item[q] < v[k];
            place[k / 2] |= r << (16 * (k % 2));
        }
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kSortK; ++k)
        if (k * NT + tid < cnt) sh.a.item[rank_of(place, k)] = v[k];
    __syncthreads();
}

// Steps 1 and 2 for particle i: the number of items, in chunks from sh.start[c] on
// in A, or -1 where a bin stays overfull.  (A function of its own:
// its registers are then not held, or spilled, through the chunks' sorts.)
__device__ __noinline__ int sort_into_chunks(const JDS J, int i, int n, float eps2, unsigned long long *A)
{
    SortShared &sh = sort_shared();
    constexpr int NT = kSortNT, kOwn = kBins / NT;   // this thread's bins
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const Side2 N = side2_neg(J.pos_hi[i], J.pos_lo[i], J.vel[i]);
    if (tid == 0) sh.cnt = 0;
    unsigned key0 = 0, place = 0;
    int shift = kBinShift, total = 0;
    auto histogram = [&](auto bin, bool first) {
        for (int q = tid; q < kBins; q += NT) sh.a.hist[q] = 0;
        __syncthreads();
        int cnt = 0;
        for (int j = tid; j < n; j += 2 * NT) {
            const uint2 key = sort_keys(J, j, j + NT, n, i, N, eps2);
            if (key.x != ~0u) atomicAdd(&sh.a.hist[bin(key.x)], 1u), ++cnt;
            if (key.y != ~0u) atomicAdd(&sh.a.hist[bin(key.y)], 1u), ++cnt;
        }
        cnt = __reduce_add_sync(kFull, cnt);
        if (lane == 0 && first) atomicAdd(&sh.cnt, cnt);
        __syncthreads();
        total = sh.cnt;
    };
    auto bin = [&](unsigned key) { return (key - key0) >> shift; };
    histogram([](unsigned key) { return key >> kBinShift; }, true);
    for (;;) {
        unsigned sum = 0, most = 0;
        for (int q = 0; q < kOwn; ++q) {
            const unsigned c = sh.a.hist[tid * kOwn + q];
            sum += c;
            most = max(most, c);
        }
        place = cta_exclusive(sum, sh.scan, lane, warp);
        if (!__syncthreads_or(most > kChunk)) break;
        // once more, over the keys' own range, if that makes the bins finer
        if (shift != kBinShift) return -1;
        unsigned lo = kBins, hi = 0;
        for (int q = tid * kOwn; q < (tid + 1) * kOwn; ++q)
            if (sh.a.hist[q]) lo = min(lo, (unsigned)q), hi = q;
        lo = __reduce_min_sync(kFull, lo);
        hi = __reduce_max_sync(kFull, hi);
        if (lane == 0) sh.lo[warp] = lo, sh.hi[warp] = hi;
        __syncthreads();
        for (int w = 0; w < kSortW; ++w) lo = min(lo, sh.lo[w]), hi = max(hi, sh.hi[w]);
        const int finer = __clz(hi - lo) - (32 - kBinBits);   // doublings of the bins
        if (finer <= 0) return -1;
        key0 = lo << kBinShift;
        shift = kBinShift - finer;
        histogram(bin, false);
    }
    for (int q = tid; q < kChunks + 2; q += NT) sh.start[q] = total;
    __syncthreads();
    // a chunk starts at the first bin that starts at or past a multiple of kChunk
    int prev = tid == 0 ? -1 : (int)((place - sh.a.hist[tid * kOwn - 1]) / kChunk);
    for (int q = 0; q < kOwn; ++q) {
        const int c = (int)(place / kChunk);   // past the last item: kChunks at most
        sh.id[tid * kOwn + q] = (unsigned char)c;
        if (c != prev && c <= kChunks) sh.start[c] = place;
        prev = c;
        place += sh.a.hist[tid * kOwn + q];
    }
    __syncthreads();
    // items to their chunk, in any order within it (the chunk's sort compares j too)
    for (int q = tid; q < kChunks + 1; q += NT) sh.next[q] = sh.start[q];
    __syncthreads();
    for (int j = tid; j < n; j += 2 * NT) {
        const uint2 key = sort_keys(J, j, j + NT, n, i, N, eps2);
        if (key.x != ~0u)
            A[atomicAdd(&sh.next[sh.id[bin(key.x)]], 1u)] = (unsigned long long)key.x << 32 | (unsigned)j;
        if (key.y != ~0u)
            A[atomicAdd(&sh.next[sh.id[bin(key.y)]], 1u)] = (unsigned long long)key.y << 32 | (unsigned)(j + NT);
    }
    __syncthreads();
    return total;
}

__global__ void __launch_bounds__(kSortNT, kSortCtas) k_force_sorted(ForceArgs fa, JDS J, SumArgs sa)
{
    static_assert(kSortNT == 256, "a thread per digit and per 32 bins");
    const int na = read_na(fa);
    if (na <= 0) return;
    SortShared &sh = sort_shared();
    __shared__ float s_res[7];
    const int n = fa.n, tid = threadIdx.x;
    const float eps2 = (float)fa.eps2;
    unsigned long long *const A = sa.scratch + (size_t)blockIdx.x * (size_t)sa.words;

    for (int a = blockIdx.x; a < na; a += gridDim.x) {
        const int i = clamp_index(fa.act[a], n);
        const int total = n <= kChunks * kChunk ? sort_into_chunks(J, i, n, eps2, A) : -1;
        float run = 0.0f;
        if (total < 0) {
            run = sa.words >= 2LL * n ? sum_in_scratch(J, i, n, eps2, A)
                                      : sum_in_scratch(J, i, n, eps2, reinterpret_cast<unsigned *>(A));
        } else {
            // 3. chunk by chunk
            for (int c = 0; c <= kChunks; ++c) {
                const int first = (int)sh.start[c], len = (int)sh.start[c + 1] - first;
                if (first >= total) break;
                if (len <= 0) continue;
                sort_chunk(sh, A + first, len);
                sum_sorted(sh, J, i, eps2, len, [&](int q) { return (int)(unsigned)sh.a.item[q]; }, run);
            }
        }
        if (tid < 7) s_res[tid] = run;
        __syncthreads();
        if (tid == 0) {
            double res[kComp];
#pragma unroll
            for (int q = 0; q < 7; ++q) res[q] = (double)s_res[q];
            store_result(fa.out, a, res);
        }
        __syncthreads();
    }
}

}  // namespace

int occupancy_sum(int mode, int *blocks_per_sm)
{
    cudaError_t e;
    if (mode == NB_SUM_FIXED)
        e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_force_fixed<kFixNT>,
                                                          kFixNT, 0);
    else if (mode == NB_SUM_FP32)
    {
        e = cudaFuncSetAttribute(k_force_seq, cudaFuncAttributeMaxDynamicSharedMemorySize, kSeqSmem);
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_force_seq, kSeqNT, kSeqSmem);
    }
    else {
        e = cudaFuncSetAttribute(k_force_sorted, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortShared));
        if (e == cudaSuccess)
            e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_force_sorted, kSortNT, sizeof(SortShared));
    }
    return e == cudaSuccess ? 0 : -1;
}

int grid_summed(const ForceArgs &fa, const SumArgs &sa)
{
    if (fa.na_dev) return sa.slots;
    const int na = fa.na_host;
    if (na <= 0) return 0;
    long long items;
    if (sa.mode == NB_SUM_FIXED)
        // one CTA per item, dealt out as CTAs end: with four warps a scheduler
        // the resident CTAs progress unevenly, and items dealt in turn left
        // 28% of the warps idle on average
        return fa.plan.p.items;
    else if (sa.mode == NB_SUM_FP32) {
        int I, T;
        seq_shape(na, sa.slots, I, T);
        items = cdiv(na, I);
    } else
        items = na;
    return (int)(items < sa.slots ? items : sa.slots);
}

int launch_force_summed(const ForceArgs &fa, const JDS &j, const SumArgs &sa, int grid,
                        cudaStream_t st)
{
    if (grid <= 0) return 0;
    if (sa.mode == NB_SUM_FIXED) {
        cudaMemsetAsync(sa.bounds, 0, 2 * sizeof(unsigned), st);
        const int gb = (int)(cdiv(fa.n, 256) < 1024 ? cdiv(fa.n, 256) : 1024);
        k_fixed_bounds<<<gb, 256, 0, st>>>(j, fa.n, sa.bounds);
        k_force_fixed<kFixNT><<<grid, kFixNT, 0, st>>>(fa, j, sa);
        long long gc = fa.na_dev ? 1024 : cdiv((long long)fa.na_host * kComp, 256);
        if (gc > 4096) gc = 4096;
        k_fixed_combine<<<(int)gc, 256, 0, st>>>(fa, sa);
        return 3;
    }
    if (sa.mode == NB_SUM_FP32) {
        k_force_seq<<<grid, kSeqNT, kSeqSmem, st>>>(fa, j, sa.slots);
        return 1;
    }
    k_force_sorted<<<grid, kSortNT, sizeof(SortShared), st>>>(fa, j, sa);
    return 1;
}

}  // namespace nbk
