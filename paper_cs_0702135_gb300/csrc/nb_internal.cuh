// nb_internal.cuh -- device data layout, control block and launchers shared by
// the CUDA translation units of the library (not part of the public ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nb.h"

namespace nbk {

constexpr int kTickBits = 40;

// Device-resident control block.  Every kernel of a block step reads its
// block time and block size from here, so a whole step can be replayed from a
// CUDA graph with no host round trip.
struct Ctrl {
    long long t_now;         // system time: block time of the last step (ticks)
    long long t_next;        // block time chosen by the scheduler (ticks)
    long long t_end;         // steps stop once the next block time would pass this
    long long steps;         // block steps taken
    long long interactions;  // sum over steps of n_active * (n - 1)
    double ekin, epot;       // last energy reduction
    int n_active;            // size of the current block; 0 = nothing to do
    int err;                 // first NB_* error raised by a kernel (0 = none)
    int err_where;           // which check raised it (for messages)
    int pad;
};

// FP64 master state, structure of arrays: x[c * n + i] for component c.
struct State {
    double *x, *v, *a, *k;   // position, velocity, acceleration, jerk
    const double *m;         // masses
    long long *t;            // particle times in ticks
    int *lev;                // block levels: dt_i = 2^-lev
    int n;
};

// j-particle records written by the predictor.
//  DS:   pos_hi = (x_hi, y_hi, z_hi, m), pos_lo = (x_lo, y_lo, z_lo, 0),
//        vel = (vx, vy, vz, 0) with x = x_hi + x_lo to 2^-48 relative.
//  FP64: pos = (x, y, z, m), vel = (vx, vy, vz, 0).
struct JDS {
    float4 *pos_hi, *pos_lo, *vel;
};
struct JF64 {
    double4_32a *pos, *vel;
};

// Force results in the public layout: acc[a][3], jerk[a][3], pot[a].
struct ForceOut {
    double *acc, *jerk, *pot;
};

// ---------------------------------------------------------------------------
// Work decomposition.  The same functions run on the host (to size buffers and
// grids) and on the device (where n_active is only known there).

#ifndef NB_IPAR_NT
#define NB_IPAR_NT 64
#endif
#ifndef NB_IPAR_R
#define NB_IPAR_R 4
#endif
#ifndef NB_IPAR_UNROLL
#define NB_IPAR_UNROLL 4
#endif

constexpr int kIparNT = NB_IPAR_NT;  // threads per CTA (= j per tile), i-parallel kernels
constexpr int kIparR = NB_IPAR_R;    // i per thread, DS i-parallel kernel
constexpr int kIparUnroll = NB_IPAR_UNROLL;  // j unrolling of the DS inner loop
#ifndef NB_IPAR_TILE_MULT
#define NB_IPAR_TILE_MULT 2
#endif
constexpr int kIparTileMult = NB_IPAR_TILE_MULT;  // DS i-parallel: j per tile = threads x this
constexpr int kIparR64 = 1;    // i per thread, FP64 i-parallel kernel
constexpr int kJparNT = 256;   // threads per CTA, j-parallel kernels
constexpr int kJparIC = 4;     // i per pass, j-parallel kernels
constexpr int kJparIC1Max = 2;  // DS j-parallel kernel: one i per pass up to this block size
constexpr int kJparMaxActive = 96;     // automatic mode, DS: j-parallel up to this block size
constexpr int kJparMaxActive64 = 32;   // automatic mode, FP64
constexpr int kIparSmallUnroll = 2;  // its j unrolling (2, 4, 8: 169, 173, 171 us for 1820 active on 65536)
constexpr int kIparSmallR = 1;      // i per thread of the small-block DS i-parallel kernel
constexpr int kSmallMaxActive = 1024;  // with a forced slice count: small-block kernel considered up to this size
constexpr int kComp = 7;       // acc xyz, jerk xyz, pot
// Clocks per j of an i-parallel CTA alone on its SM, and of each CTA with the SM full, for the
// four-i and the one-i kernel, and how many are resident (see fine_cost).
constexpr unsigned kFineAlone4 = 200, kFineEach4 = 95, kFineRes4 = 4;
constexpr unsigned kFineAlone1 = 105, kFineEach1 = 22, kFineTail1 = 50, kFineRes1 = 16;
constexpr unsigned kFineItemJ = 32;
constexpr int kFineMaxActive = 20000;

struct Plan {
    int n_iblk;   // i-blocks (i-parallel) or i-chunks (j-parallel)
    int S;        // j slices of a sliced i-block
    int jslice;   // j per slice (multiple of the tile)
    int items;    // work items: n_whole + (n_iblk - n_whole) * S
    int n_whole;  // i-parallel: leading i-blocks taken whole (all j in one item, result
                  // written directly); the others are sliced.  0 for uniform plans.
    int a0;       // first block position of the sliced i-blocks (n_whole * i-block size)
};

__host__ __device__ inline int cdiv(long long a, long long b) { return (int)((a + b - 1) / b); }

// i-parallel: CTAs own iblk consecutive active particles and one j slice.
// The slice count S starts at s0 = 1, or, with fewer than two i-blocks per
// resident CTA, at the count that makes two; then among a few candidates
// (s0 .. s0 + 7 and the counts that fill 1 .. 8 waves of the slots resident
// CTAs exactly) the smallest whose last wave is at least 95% full is taken,
// else the one with the fullest last wave.  Slices keep at least two tiles and
// the partials fit in part_cap doubles.  Integer arithmetic only, computed
// once per force launch (host or scheduler, see ForcePlan).
// Every quotient in the slice search has operands below 2^31 (item counts are
// at most 8 slots + 8 i-blocks), so it uses 32-bit unsigned divisions, which
// cost a fraction of the 64-bit ones.
__host__ __device__ inline unsigned udiv(unsigned a, unsigned b) { return a / b; }
__host__ __device__ inline unsigned ucdiv(unsigned a, unsigned b) { return (a + b - 1) / b; }

__host__ __device__ inline bool better_fill(unsigned items_a, unsigned slots, unsigned items_b)
{
    // fill(x) = x / (ceil(x / slots) * slots); compare fill(a) > fill(b)
    const unsigned long long wa = ucdiv(items_a, slots), wb = ucdiv(items_b, slots);
    return items_a * wb > items_b * wa;
}

__host__ __device__ inline bool fill_ok(unsigned items, unsigned slots)
{
    const unsigned long long w = ucdiv(items, slots);
    return 20ULL * items >= 19ULL * w * slots;
}

// Cost of one plan shape in j per resident CTA: waves of `items` equal items
// of `len` j each on `slots` CTAs, with a per-item overhead worth
// kItemCostJ j (the i records, the tile start-up and the result stores).
constexpr unsigned kItemCostJ = 64;
__host__ __device__ inline unsigned long long wave_cost(unsigned items, unsigned slots, unsigned len)
{
    return (unsigned long long)ucdiv(items, slots) * (len + kItemCostJ);
}

__host__ __device__ inline unsigned slice_len(int n, int S, int tile)
{
    return (unsigned)cdiv(cdiv(n, S), tile) * (unsigned)tile;
}

__host__ __device__ inline unsigned ugcd(unsigned a, unsigned b)
{
    while (b) {
        const unsigned t = a % b;
        a = b;
        b = t;
    }
    return a;
}

__host__ __device__ inline Plan plan_ipar(int na, int n, int iblk, int tile, int slots,
                                          int split, long long part_cap, bool tail_split = false)
{
    Plan p;
    p.n_iblk = (int)ucdiv((unsigned)na, (unsigned)iblk);
    p.n_whole = 0;
    p.a0 = 0;
    const int smax_tiles = (int)ucdiv((unsigned)n, 2u * (unsigned)tile);
    const long long pmax = part_cap / ((long long)kComp * (na > 0 ? na : 1));
    int smax = smax_tiles < pmax ? smax_tiles : (int)pmax;
    if (smax < 1) smax = 1;
    int S;
    if (split > 0) {
        S = split < smax ? split : smax;
    } else {
        const unsigned nib = (unsigned)p.n_iblk, us = (unsigned)slots;
        int s0 = nib >= 2 * us ? 1 : (int)ucdiv(2 * us, nib);
        if (s0 > smax) s0 = smax;
        int best = s0, first_ok = fill_ok(nib * (unsigned)s0, us) ? s0 : 0;
#pragma unroll
        for (int q = 0; q < 24; ++q) {
            int s;
            if (q < 8) s = s0 + q;
            else if (q < 16) s = (int)udiv((unsigned)(q - 7) * us, nib);
            else s = (int)ucdiv((unsigned)(q - 15) * us, nib);
            if (s < s0 || s > smax) continue;
            const unsigned it = nib * (unsigned)s;
            if (fill_ok(it, us) && (first_ok == 0 || s < first_ok)) first_ok = s;
            if (better_fill(it, us, nib * (unsigned)best)) best = s;
        }
        S = first_ok ? first_ok : best;
        // With at least one full wave of i-blocks, the blocks of the full
        // waves may instead run whole and only the remainder be sliced, in a
        // slice count that fills its waves (multiples of slots / gcd(rem,
        // slots) fill them exactly): taken when its cost is lower.
        const unsigned rem = nib % us;
        if (tail_split && nib >= us && rem > 0) {
            const unsigned whole = nib - rem;
            const long long arem = (long long)na - (long long)whole * iblk;
            const long long pmax_t = part_cap / ((long long)kComp * arem);
            int smax_t = smax_tiles < pmax_t ? smax_tiles : (int)pmax_t;
            const unsigned long long c_uni = wave_cost(nib * (unsigned)S, us, slice_len(n, S, tile));
            const unsigned long long c_whole = wave_cost(whole, us, (unsigned)n);
            const unsigned per = us / ugcd(rem, us);
            int bt = 0;
            unsigned long long c_best = c_uni;
#pragma unroll
            for (int q = 0; q < 12; ++q) {
                const int s = q < 4 ? (int)(per * (unsigned)(q + 1)) : (int)ucdiv((unsigned)(q - 3) * us, rem);
                if (s < 2 || s > smax_t) continue;
                const unsigned long long c =
                    c_whole + wave_cost(rem * (unsigned)s, us, slice_len(n, s, tile));
                if (c < c_best) {
                    c_best = c;
                    bt = s;
                }
            }
            if (bt > 0) {
                p.n_whole = (int)whole;
                p.a0 = (int)((long long)whole * iblk);
                S = bt;
            }
        }
    }
    p.jslice = (int)slice_len(n, S, tile);
    p.S = cdiv(n, p.jslice);
    p.items = p.n_whole + (p.n_iblk - p.n_whole) * p.S;
    return p;
}

// Work item w of an i-parallel plan: its i-block ib, j range [j0, j1) and
// slice sl (-1 for an i-block taken whole, whose result is final).
__host__ __device__ inline void ipar_item(int w, int n_iblk, int n_whole, int S, int jslice, int n,
                                          int &ib, int &sl, int &j0, int &j1)
{
    if (w < n_whole || S == 1) {
        ib = w;
        sl = -1;
        j0 = 0;
        j1 = n;
    } else {
        const int nb = n_iblk - n_whole, q = w - n_whole;
        ib = n_whole + q % nb;
        sl = q / nb;
        j0 = sl * jslice;
        j1 = n < j0 + jslice ? n : j0 + jslice;
    }
}

// j-parallel: CTAs own ic active particles and one j slice; each thread takes
// every nt-th j of the slice, at least eight per thread.  The slice count aims
// at two work items per resident CTA, else (slices too short) at one, so that
// the last wave is not a small remainder.
__host__ __device__ inline Plan plan_jpar(int na, int n, int nt, int ic, int slots,
                                          long long part_cap)
{
    Plan p;
    p.n_iblk = cdiv(na, ic);
    int S = cdiv(2LL * slots, p.n_iblk);
    const int smax = cdiv(n, 8LL * nt);
    if (S > smax) S = cdiv((long long)slots, p.n_iblk);
    if (S > smax) S = smax;
    long long pmax = part_cap / ((long long)kComp * ic * p.n_iblk);
    if (S > pmax) S = (int)pmax;
    if (S < 1) S = 1;
    p.jslice = cdiv(cdiv(n, S), nt) * nt;
    p.S = cdiv(n, p.jslice);
    p.items = p.n_iblk * p.S;
    p.n_whole = 0;
    p.a0 = 0;
    return p;
}

// Lanes per output of the slice combine: a power of two T <= 32, T <= S, with
// about 2^18 threads in all (T * 7 na), so that both small blocks with many
// slices and large blocks with few get enough loads in flight.
__host__ __device__ inline int combine_lanes(int na, int S)
{
    const long long want = (1LL << 18) / ((long long)kComp * (na > 0 ? na : 1));
    int T = 1;
    while (T < 32 && T < want && 2 * T <= S) T *= 2;
    return T;
}

// Which kernel serves a block of na particles: jpar for na <= jpar_max.
__host__ __device__ inline bool use_jpar(int na, int jpar_max) { return na <= jpar_max; }

// Force kernels by block size: j-parallel, small-block i-parallel (one i per
// thread, blocks of kIparNT i), i-parallel (kIparR i per thread, blocks of
// kIparNT * kIparR i).  Where the rule below on fine plans does not apply (a
// forced slice count), the small-block kernel serves a block when its padded
// i count is at most 3/4 of the other's: up to 192, 257..384 and 513..576
// active with 64-i and 256-i blocks.  small_max <= jpar_max disables it.
__host__ __device__ inline bool small_pays(int na)
{
    const long long s = (long long)cdiv(na, kIparNT) * kIparNT;
    const long long r = (long long)cdiv(na, kIparNT * kIparR) * (kIparNT * kIparR);
    return 4 * s <= 3 * r;
}

enum Regime { kRegJpar = 0, kRegSmall = 1, kRegIpar = 2 };
__host__ __device__ inline int regime_of(int na, int jpar_max, int small_max)
{
    if (na <= jpar_max) return kRegJpar;
    if (na <= small_max && small_pays(na)) return kRegSmall;
    return kRegIpar;
}

// DS i-parallel, up to kFineMaxActive active: kernel and slice length are
// chosen together, by the time of the busiest SM.  Candidate c: the four-i
// (c < 16) or the one-i kernel, with the slice length in tiles that makes
// c % 16 + 1 waves of its resident CTAs (a single tile where that is already
// less than a wave).  Four-i items go to the CTAs in turn: an SM given m items
// runs `res` at a time, k together at max(alone, k each) clocks per j (one
// CTA alone cannot hide its latencies).  One-i items are taken as CTAs end
// (with four warps a scheduler, CTAs progress unevenly): each clocks per j and
// item on average, and a tail.  Every item costs kFineItemJ j more.  Both
// kernels sum the same 128-j tiles in the same order, so the choice does not
// show in the tile partials.
//
// The one-i kernel reaches 90% of the four-i kernel's rate on full blocks,
// pads the block to 64 instead of 256 and cuts it four times as fine, so it
// wins wherever the padding or a part-filled GPU costs the other more than a
// tenth.  Force and combine, us, four-i plan before / this rule: 256 active
// on 256 bodies 42 / 17, 1024 on 1024 44 / 17, 4096 on 4096 49 / 40, 300 on
// 4096 25 / 19; on 65536: 700 100 / 79, 1820 208 / 165, 4096 347 / 330, 8192
// 654 / 625, 20000 1579 / 1475.  Above kFineMaxActive the two are within 2%
// and plan_ipar's search, which also runs blocks whole, is kept.
constexpr int kFineCands = 32;
__host__ __device__ inline unsigned fine_clocks(unsigned m, unsigned res, unsigned alone, unsigned each)
{
    const unsigned rem = m % res;
    unsigned t = m / res * (res * each);
    if (rem) t += rem * each > alone ? rem * each : alone;
    return t;
}

// Slice length in tiles of candidate c.
__host__ __device__ inline unsigned fine_tiles(int na, int n, int sms, int c)
{
    const bool one = c >= 16;
    const unsigned tiles = ucdiv((unsigned)n, (unsigned)(kIparNT * kIparTileMult));
    const unsigned nib = ucdiv((unsigned)na, (unsigned)(kIparNT * (one ? kIparSmallR : kIparR)));
    const unsigned slots = (unsigned)sms * (one ? kFineRes1 : kFineRes4) * (unsigned)(c % 16 + 1);
    return (unsigned)(((unsigned long long)tiles * nib + slots - 1) / slots);
}

// Relative time of candidate c for na active on n (~0: not possible).
__host__ __device__ inline unsigned long long fine_cost(int na, int n, int sms, long long part_cap, int c)
{
    const bool one = c >= 16;
    const unsigned tile = (unsigned)(kIparNT * kIparTileMult), L = fine_tiles(na, n, sms, c);
    const unsigned nib = ucdiv((unsigned)na, (unsigned)(kIparNT * (one ? kIparSmallR : kIparR)));
    const unsigned S = ucdiv(ucdiv((unsigned)n, tile), L);
    if (S > 1 && (long long)S * kComp * na > part_cap) return ~0ULL;
    const unsigned items = nib * S;
    unsigned t;
    if (one) {
        t = (unsigned)((unsigned long long)items * kFineEach1 / (unsigned)sms) + kFineTail1;
        if (t < kFineAlone1) t = kFineAlone1;
    } else {
        t = fine_clocks(ucdiv(items, (unsigned)sms), kFineRes4, kFineAlone4, kFineEach4);
    }
    return (unsigned long long)(L * tile + kFineItemJ) * t;
}

// The work decomposition of one force launch: the block size, the kernel
// that serves it and that kernel's plan.  It is computed once per launch, by
// make_force_plan on the host when the block size is known there, else by the
// scheduler's last thread next to the block size; kernels read it instead of
// planning in every CTA.
struct ForcePlan {
    Plan p;        // plan of the serving kernel (zero for the FP32 summation variants)
    int na;        // block size
    int regime;    // kRegJpar / kRegSmall / kRegIpar (summation variants: kRegIpar)
    int ic;        // j-parallel: i per pass
    int lanes;     // slice combine: lanes per output
};

// Everything a force launch needs.
struct ForceArgs {
    int n;                    // j count
    const int *act;           // active indices (device)
    const int *na_dev;        // device block size, or nullptr to use na_host
    int na_host;
    ForcePlan plan;           // the plan for na_host (na_dev == nullptr)
    const ForcePlan *plan_dev;  // the plan for *na_dev, written by the scheduler
    int precision;            // NB_DS or NB_FP64
    int summation;            // NB_SUM_*
    int slots_sum;            // resident CTAs of the summation variant's kernel
    int jpar_max;             // regime boundaries (see regime_of)
    int small_max;
    int split;                // forced slice count for i-parallel, 0 = auto
    int slots_ipar, slots_jpar, slots_small;
    int sms;                  // SMs of the device (0: no fine plans)
    long long part_cap;       // capacity of part in doubles
    double *part;             // slice partials: part[(s * 7 + c) * na + a]; the DS
                              // j-parallel kernel: part[(chunk * 7 ic + e) * S + s]
    int *work;                // device-sized launches: items taken by the one-i kernel's CTAs
                              // beyond their first (zeroed by the scheduler)
    int *jcnt;                // per-chunk slice arrival counters (zero between launches)
    ForceOut out;
    double eps2;
    int *err;                 // device error word
};

// Summation variants (k_sum.cu): the force with single-precision pair terms in
// IEEE round-to-nearest arithmetic, summed in 64-bit fixed point (GRAPE-style,
// independent of summation order), or in FP32 in index order, or in FP32
// smallest pair force first.
struct SumArgs {
    int mode;                       // NB_SUM_FIXED, NB_SUM_FP32 or NB_SUM_FP32_SORTED
    unsigned *bounds;               // [2] fixed point: largest fl32 mass, largest fl32 |vx|+|vy|+|vz| (bits)
    unsigned long long *scratch;    // sorted: `words` per resident CTA (sort_scratch_size)
    long long words;
    int slots;                      // resident CTAs of the mode's force kernel
};
constexpr int kFixNT = 64;   // fixed point: threads per CTA, one i each (slices: multiples of it)
// fixed point: CTAs per SM the registers are held to (8, 9, 10, 12: 13.29, 13.23, 13.22, 13.36 ms
// on 65536 bodies all active)
constexpr int kFixCtas = 10;
// fixed point: blocks of at least an eighth of the slots in i-blocks plan as if there were this
// many times the slots, so that the items are short against the launch (1, 2, 4: 13.45, 13.45,
// 13.29 ms); smaller blocks have too few j a slice for it (with and without, ms on 65536
// bodies: 12288 active 2.55 and 2.59, 8192 1.75 and 1.79, 4096 0.90 and 0.93, 1820 0.48 and
// 0.45: the two meet somewhat below the line)
constexpr int kFixWaves = 4;
constexpr int kSeqNT = 640;         // FP32 index order: threads per CTA
constexpr int kSortNT = 256;        // FP32 sorted: one CTA per i
constexpr int kSortCtas = 4;        // and at least this many per SM
constexpr int kChunk = 2048, kChunks = 255;   // items aimed at in a chunk, and how many chunks at most

// FP32 sorted: 8-byte words of scratch of a CTA (n keyed items; twice that where
// every block takes the sort of all items, which moves them between two
// arrays), and the CTAs.  All that fit the SMs (1820 active on 65536 bodies:
// 5.1 ms with four an SM, 18.6 ms with a single larger one) unless their scratch is
// more than a 32nd of the free memory, or 4 GiB: then as many as 16 n bytes an SM
// hold, which is what one CTA an SM with two arrays takes.
struct SortScratch {
    long long words;
    int slots;
};
inline SortScratch sort_scratch_size(long long n, int sms, int per_sm, unsigned long long free_bytes)
{
    SortScratch r;
    r.words = n <= (long long)kChunks * kChunk ? n : 2 * n;
    const long long part = (long long)(free_bytes / 32), least = 16 * n * sms, cap = 4LL << 30;
    long long bytes = part > least ? part : least;
    if (bytes > cap) bytes = cap;
    const long long fit = bytes / (8 * r.words), all = (long long)sms * per_sm;
    r.slots = (int)(fit < 1 ? 1 : (fit < all ? fit : all));
    return r;
}
constexpr int kErrFixedScale = 64;  // device error word: fixed-point scales out of range
constexpr int kErrInput = 65;       // device error word: a non-finite value or a negative mass

// Whether a block of na is planned by fine_cost (also a larger one whose
// four-i items of one tile are less than a wave), and its cheapest candidate.
__host__ __device__ inline bool fine_applies(const ForceArgs &fa, int na)
{
    return fa.sms > 0 && fa.precision == NB_DS && fa.summation == NB_SUM_COMPENSATED && fa.split == 0 &&
           na > fa.jpar_max &&
           (na <= kFineMaxActive ||
            (long long)cdiv(fa.n, kIparNT * kIparTileMult) * cdiv(na, kIparNT * kIparR) <= fa.slots_ipar);
}
__host__ __device__ inline int fine_best(const ForceArgs &fa, int na)
{
    unsigned long long best = ~0ULL;
    int bc = -1;
    for (int c = 0; c < kFineCands; ++c) {
        const unsigned long long t = fine_cost(na, fa.n, fa.sms, fa.part_cap, c);
        if (t < best) best = t, bc = c;
    }
    return bc;
}

// fine: the cheapest fine candidate where fine_applies, found by the caller
// (the scheduler's warp evaluates all candidates at once); -2 = find it here.
__host__ __device__ inline ForcePlan make_force_plan(const ForceArgs &fa, int na, int fine = -2)
{
    ForcePlan f{};
    f.na = na;
    f.regime = kRegIpar;
    if (na <= 0) return f;
    if (fa.summation == NB_SUM_FIXED) {
        f.p = plan_ipar(na, fa.n, kFixNT, kFixNT,
                        fa.slots_sum * (8LL * cdiv(na, kFixNT) >= fa.slots_sum ? kFixWaves : 1), fa.split, fa.part_cap / 2);
        return f;
    }
    if (fa.summation != NB_SUM_COMPENSATED) return f;   // no slices
    const bool f64 = fa.precision == NB_FP64;
    if (fine == -2) fine = fine_applies(fa, na) ? fine_best(fa, na) : -1;
    if (fine >= 0) {
        const bool one = fine >= 16;
        f.regime = one ? kRegSmall : kRegIpar;
        f.p.n_iblk = cdiv(na, kIparNT * (one ? kIparSmallR : kIparR));
        f.p.jslice = (int)fine_tiles(na, fa.n, fa.sms, fine) * kIparNT * kIparTileMult;
        f.p.S = cdiv(fa.n, f.p.jslice);
        f.p.items = f.p.n_iblk * f.p.S;
        f.lanes = combine_lanes(na, f.p.S);
        return f;
    }
    f.regime = f64 ? (use_jpar(na, fa.jpar_max) ? kRegJpar : kRegIpar)
                   : regime_of(na, fa.jpar_max, fa.small_max);
    if (f.regime == kRegJpar) {
        f.ic = !f64 && na <= kJparIC1Max ? 1 : kJparIC;
        f.p = plan_jpar(na, fa.n, kJparNT, f.ic, fa.slots_jpar, fa.part_cap);
    } else {
        const int r = f64 ? kIparR64 : (f.regime == kRegSmall ? kIparSmallR : kIparR);
        const int slots = f.regime == kRegSmall ? fa.slots_small : fa.slots_ipar;
        f.p = plan_ipar(na, fa.n, kIparNT * r, kIparNT * (f64 ? 1 : kIparTileMult), slots, fa.split,
                        fa.part_cap, true);
    }
    f.lanes = combine_lanes(na - f.p.a0, f.p.S);
    return f;
}

#ifdef __CUDACC__
// The plan of this launch (a uniform load for the device-sized launches).
__device__ __forceinline__ ForcePlan load_plan(const ForceArgs &fa)
{
    return fa.plan_dev ? *fa.plan_dev : fa.plan;
}
#endif

// Persistent block-step loop (k_run.cu): nb_run in one cooperative launch for
// systems of up to kRunMaxN particles, kRunNT threads per CTA, one CTA per
// `per` particles.
constexpr int kRunNT = 256;
// a CTA corrects up to this many particles of a step with four lanes each
constexpr int kRunQuadMax = 16;
constexpr int kRunMaxN = 16384;   // above it the per-stage graph, using every SM for the force, is faster
constexpr int kRunIndexBits = 14;   // particle index in a block record's tag, below the step
constexpr int kRunPerLane = 8;      // CTAs at most: 32 times this
// steps per launch at most: a tag's step number must not come round again
constexpr long long kRunMaxSteps = 1LL << 17;
// Steps of nb_run's next launch or batch: of the max_steps from counter value steps0
// on, those that are left at counter value `steps`, whoever took the others.
inline long long run_batch(long long max_steps, long long steps0, long long steps, long long limit)
{
    const long long left = max_steps - (steps - steps0);
    return left < limit ? left : limit;
}
static_assert(kRunMaxN == 1 << kRunIndexBits && kRunMaxSteps < 1LL << (32 - kRunIndexBits), "tags");
struct RunArgs {
    State s;
    JDS j;
    Ctrl *ctrl;
    int n, ncta, per;            // particles, CTAs, particles per CTA (<= kRunNT)
    float eps2f;                 // single-precision eps^2 of the pair terms
    double eta;
    int level_min, level_fixed;
    long long t_end, max_steps;  // stop before a block time past t_end, or after max_steps steps
    int *act;                    // [n] block list (written at the end)
    // exchanged between CTAs, all zero at launch:
    ulonglong2 *minrec;          // [2][ncta] least end time; count, error bit and step
    ulonglong2 *maxrec;          // [2][ncta] fixed point: mass and |v|_1 bounds (float bits), step
    unsigned long long *flag;    // [ncta] steps whose partials are written
    float4 *blk;                 // [n][3] block records: hi, lo, velocity, each with its tag
    double *part;                // [n][ncta][8] partials (fixed point: pairs of int64, [16])
};

// Reverse mode (k_adjoint.cu).  Force-VJP records: DS (x_hi, y_hi, z_hi, m),
// (x_lo, y_lo, z_lo, 0), (vx, vy, vz, 0), (abar, 0), (kbar, 0); FP64 (x, y,
// z, m), (v, 0), (abar, 0), (kbar, 0).
struct VjpRec {
    float4 ph, pl, v, ab, kb;
};
struct VjpRecDS {
    float4 *ph, *pl, *v, *ab, *kb;
};
struct VjpRec64 {
    double4_32a *x, *v, *ab, *kb;
};
struct VjpArgs {
    int n;
    double eps2;
    int slots;
    long long part_cap;
    Plan plan;             // over all n particles (set by the launcher)
    double *part;          // slice partials part[(s * 7 + c) * n + k]
    VjpRecDS rec;
    VjpRec64 rec64;
    const double *m;
    double *xbar, *vbar, *mbar;  // outputs [n][3], [n][3], [n] (overwritten)
};

// One kernel of a trajectory with a shared step 2^-level (k_shared_step).
enum ShMode { kShPredict = 0, kShStart = 1, kShCorrect = 2 };
struct SharedStep {
    int mode;              // predict only; take the force as acc and jerk; correct with it
    bool predict;          // then write the next step's j records
    State src, dst, copy;  // state before and after the step; copy.x may be null
    int level, precision;
    // the force: slices part[(s * 7 + c) * (n - a0) + (a - a0)] from particle a0 on
    // when S > 1, the results themselves otherwise
    const double *part;
    int S, a0;
    ForceOut out;
    JDS jds;
    JF64 jf;
};

// One kernel of its reverse pass (k_adj_step).
enum AdjMode { kAdjNone = 0, kAdjPre = 1, kAdjInitial = 2 };
struct AdjStep {
    bool post, add;        // take the VJP through the predictor, or just add it
    int pre;               // then the records of the next VJP
    State st;              // the state those start from
    int level, precision, S;
    const double *part;    // S > 1: the VJP's slices, else xg, vg, mg
    const double *xg, *vg, *mg;
    double *xb, *vb, *ab, *kb, *mb;
    VjpRecDS rec;
    VjpRec64 rec64;
};

// ---------------------------------------------------------------------------
// Launchers (defined in the .cu files).

// k_force.cu
// Returns the number of kernels launched.
// combine: add the slices of an i-parallel launch (else the caller does).
int launch_force_ds(const ForceArgs &fa, const JDS &j, bool softened, int grid_ipar, int grid_jpar,
                    int grid_small, bool combine, cudaStream_t st);
void launch_force_f64(const ForceArgs &fa, const JF64 &j, bool softened, int grid_ipar,
                      int grid_jpar, cudaStream_t st);
int occupancy_force(int precision, int regime, int *blocks_per_sm);

// k_sum.cu
int occupancy_sum(int mode, int *blocks_per_sm);
int grid_summed(const ForceArgs &fa, const SumArgs &sa);
int launch_force_summed(const ForceArgs &fa, const JDS &j, const SumArgs &sa, int grid,
                        cudaStream_t st);

// k_run.cu
int run_layout(int n, int sms, int blocks_per_sm, int *ncta, int *per);
int occupancy_run(int summation, int *blocks_per_sm);
cudaError_t launch_run(const RunArgs &ra, int summation, cudaStream_t st);
cudaError_t launch_check_wait(const unsigned long long *counter, long long limit_cycles, Ctrl *ctrl,
                              cudaStream_t st);

// k_step.cu
void launch_predict(const State &s, long long t_val, const long long *t_ptr, const int *gate,
                    int precision, JDS jds, JF64 jf, cudaStream_t st);
// Blocks of at most kCorrectQuadPerSM x SMs particles are corrected with four
// lanes per particle (correct_particle_quad), larger ones one thread each.
constexpr int kCorrectQuadPerSM = 16;
void launch_correct(const State &s, const int *act, int na_host, const int *na_dev,
                    long long t_val, const long long *t_ptr, const double *acc_new,
                    const double *jerk_new, double eta, int level_min, int level_fixed,
                    int *err, int sms, cudaStream_t st);
void launch_initial_steps(const State &s, const double *acc, const double *jerk, double eta_init,
                          int level_min, int level_fixed, int *err, cudaStream_t st);
// Also writes the plan of the force on the new block (make_force_plan(fa, n_active))
// and predicts every particle to the block time into the j records (as
// launch_predict), unless no block is left before the end time.
void launch_schedule(const State &s, Ctrl *ctrl, long long *blockmin, int *blockcnt, int *act,
                     int nblocks, const ForceArgs &fa, ForcePlan *plan_out, int precision,
                     const JDS &jds, const JF64 &jf, cudaStream_t st);
int schedule_blocks(int n);
void launch_energy(const State &s, const long long *t_ptr, const double *pot, double *part,
                   Ctrl *ctrl, cudaStream_t st);
int energy_blocks(int n);
void launch_validate(const int *idx, int na, int n, unsigned int *bitmap, int *err,
                     cudaStream_t st);
// na > 0 results from res to out (see k_publish); validate: check idx[na] first.
constexpr int kPublishCheckMax = 1024;
struct PublishArgs {
    ForceOut res, out;
    int na, n;
    const int *idx;
    bool validate;
    Ctrl *ctrl, *host;
};
void launch_publish(const PublishArgs &p, cudaStream_t st);
void launch_gather_state(const State &s, double *x, double *v, double *a, double *k,
                         cudaStream_t st);
void launch_scatter_state(const State &s, const double *x, const double *v, const double *a,
                          const double *k, cudaStream_t st);
void launch_iota(int *p, int n, cudaStream_t st);
// Raises kErrInput unless every value of p[cnt] is finite (and, with
// nonneg, >= 0).
void launch_check_input(const double *p, long long cnt, bool nonneg, int *err, cudaStream_t st);

// k_adjoint.cu
int vjp_slots(int precision, int sms);
int launch_force_vjp(const VjpArgs &va, int precision, bool softened, bool combine, int *slices,
                     cudaStream_t st);
void launch_shared_step(const SharedStep &q, cudaStream_t st);
void launch_shared_done(const State &s, Ctrl *ctrl, int *act, long long steps, int level, cudaStream_t st);
void launch_shared_times(const State &s, long long t, int level, cudaStream_t st);
void launch_adj_step(const AdjStep &q, cudaStream_t st);
void launch_adj_pre(const State &s, double dt, const double *xb, const double *vb, double *ab,
                    double *kb, int precision, const VjpRecDS &rec, const VjpRec64 &rec64,
                    cudaStream_t st);
void launch_adj_post(int n, double dt, double *xb, double *vb, double *ab, double *kb, double *mb,
                     const double *xg, const double *vg, const double *mg, cudaStream_t st);
void launch_adj_initial_rec(const State &s, const double *ab, const double *kb, int precision,
                            const VjpRecDS &rec, const VjpRec64 &rec64, cudaStream_t st);
void launch_add3(int n, double *dst, const double *src, double *dst2, const double *src2,
                 double *dstm, const double *srcm, cudaStream_t st);
void launch_set_ak(const State &s, const double *acc, const double *jerk, cudaStream_t st);
void launch_copy_state(const State &dst, const State &src, cudaStream_t st);

}  // namespace nbk
