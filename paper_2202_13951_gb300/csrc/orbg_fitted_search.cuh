/*
 * orbg_fitted_search.cuh -- full ORBGRAND with a piece-wise linear model
 * fitted to each block (Sec. III-E), searched in that block's own order
 * (Sec. III-D).
 *
 * Per block, in four launches (each kernel's code stays small enough for
 * the instruction cache: in one fused kernel the fit's double-precision code
 * and the search's tree walk, run by different warps of an SM at once, made
 * instruction fetch the largest stall).  The first launch does steps 1-3
 * and finishes the blocks that need no search; the second takes the others
 * from an open list, with their order and model in a handover record, one
 * warp per block; a block whose search grows long there goes to the third,
 * where all warps of a CTA search it by pair look-ups (orbg_fitpair_kernel);
 * the few that one does not cover (weights past its counting table, too many
 * patterns tied at the hit's weight, an order of fewer patterns than the cap)
 * go to the fourth, where a CTA walks the whole tree:
 *   1. load, hard decision y, starting syndrome s0 = H y (as the other
 *      decoders: load_block);
 *   2. the exact reliability order pi (sort_block) and the ordered curve
 *      L_1 <= ... <= L_n;
 *   3. the fit: anchors by the largest chord gap (every lane takes a share of
 *      the indices; the warp keeps the largest gap, the smaller index on
 *      ties), then Eq. Q and Eq. quant on one lane (orbg_fit.cuh, the same
 *      double operations as the oracle);
 *   4. the integer weight rho_j of every sorted position j (Eq. relest_seg:
 *      J_{i-1} + beta_i (j - I_{i-1}) on segment i) and the suffix minima
 *      msuf_j = min over j' >= j of rho_j';
 *   5. the search for the first code-book member in the order of increasing
 *      reliability weight R(z) = sum of rho over the flipped positions, ties
 *      by Hamming weight and then positions lexicographically (the order
 *      every decoder of this library uses inside one weight).
 *
 * The search walks the subsets of {1..n} as a binary tree in lexicographic
 * order: node S = {j_1 < ... < j_t} has the child S + {j_t + 1} ("add") and
 * the next sibling S - {j_t} + {j_t + 1} ("replace"); every non-empty subset
 * is reached once from the root {1}.  Everything below a node keeps
 * j_1..j_{t-1} and adds positions >= j_t, so R(S) - rho_{j_t} + msuf_{j_t}
 * bounds the weight of the node and all it leads to from below; a pass with
 * bound Rhi enters only nodes whose bound is <= Rhi and tests those with
 * R <= Rhi (the weights rho need not increase with j).  The 32 lanes of the
 * warp each walk a part of the tree depth first (lane l starts with the sets
 * whose least position is l + 1), with their positions on a per-lane stack
 * in shared memory; a lane that runs out of work is given the "replace"
 * branch of a lane that is about to take its "add" branch; a lane at a leaf
 * also tests up to kLeafRun of the leaf's later siblings in the same step
 * while they are leaves too (the lanes stay in step: a longer inner run
 * would hold the other lanes).  When the warps of a CTA share a block, in
 * the third and fourth launch, the tree is cut into kClasses classes by the sets' second positions (modulo
 * kClasses; the singletons by their position), the warps take classes from
 * a counter, and each pass's node counts and least member are combined over
 * the warps.
 *
 * Passes run with growing bounds ("bands"): a pass that finds code-book
 * members lowers its bound to the lightest one found, and the least of
 * them in the order (weight, Hamming weight, positions) is the decoding; a
 * second pass over the nodes up to that weight counts the patterns that
 * come before it, which gives its query index.  A pass without a member
 * that already covers `cap` queries ends the block as abandoned.  Every
 * pass is a finite walk of a finite tree; each also stops after a fixed
 * number of steps (a guard, never reached by a correct walk) and marks the
 * block ORBG_BLOCK_RANGE, as does a search that would need weights beyond
 * 2^26 - 1.
 */
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "orbg_decode_block.cuh"
#include "orbg_fit.cuh"

namespace orbg_fitsearch {

using namespace orbg_dev;

constexpr int kWarps = 8;                   /* warps per CTA, one block each */
constexpr int kDepth = 31;                  /* largest pattern the stack holds */
constexpr uint32_t kRhoInf = 1u << 30;      /* weight of a position never reached */
constexpr int32_t kRmax = (1 << 26) - 1;    /* heaviest reliability weight searched */
constexpr int kLeafRun = 3;                /* leaf siblings tested per step besides the node */
/* Nodes a one-warp pass may test before a CTA takes over (a quarter of the
 * cap if less): kSplit, or kSplitSmall where a batch has at most two blocks a
 * resident warp and the CTAs wait for work.  Measured, us a call, three lines,
 * 100,000 BCH(127,113) and 20,000 CA-Polar[256,234] blocks, and 3,000 BCH
 * blocks of two lines: 256 1,415, 1,473 and 223; 512 1,361, 1,353 and 242;
 * 1024 1,340, 1,386 and 330.  (A pass tests about four times as many as
 * the one before, from 70 on.)
 * kSplitFew in a batch of so few positions that
 * its longest search mostly ends there, where a CTA's takes 60 us more for a
 * single block: up to kFewPositions, and past 14 parity bits, where a hit by
 * chance does not end a long search, up to kFewBlocks.  One and three lines,
 * us, 256 / 1024 / no handover: BCH 100 blocks 120, 122 / 94, 116 / 94, 115,
 * 300 blocks 151, 154 / 95, 117 / 95, 116, 1,000 blocks 157, 166 / 234, 263 /
 * 1,614, 860; a (256,244) code 10 blocks 162, 170 / 139, 148 / 140, 149, 300
 * blocks 212, 210 / 315, 286 / 492, 526; CA-Polar[256,234] 10 blocks 89, 184 /
 * 89, 124 / 89, 125, 100 blocks 199, 204 / 240, 267 / 1,891, 348. */
constexpr uint32_t kSplit = 512;
constexpr uint32_t kSplitSmall = 256;
constexpr uint32_t kSplitFew = 1024;
constexpr int64_t kFewPositions = 38912; /* 128 for two blocks an SM */
constexpr int64_t kFewBlocks = 32;
constexpr int32_t kNoHit = 0x7FFFFFFF;
constexpr int kBlockRange = ORBG_BLOCK_RANGE; /* abandoned[] value: beyond the search range */

/* Shared memory of one warp (one block in flight). */
template <int W> struct FsSmem {
    typedef typename Syn<W>::T T;
    uint32_t *rho;   /* [258] rho_j, j = 1..n; rho[n + 1] = kRhoInf */
    uint32_t *msuf;  /* [258] suffix minima, msuf[n + 1] = kRhoInf */
    uint32_t *c0;    /* [258] first syndrome word of position j; c0[0] = 0 */
    T *h;            /* [258] whole syndrome of position j (W > 1) */
    float *L;        /* [256] ordered reliabilities */
    uint8_t *pi;     /* [256] received index of sorted position j - 1 */
    uint8_t *cw;     /* [256] staged codeword */
    uint8_t *stk;    /* [32][32] stk[d * 32 + lane]: j_{d+1} of the lane's node */
    uint8_t *hb;     /* [32][32] hb[i * 32 + lane]: the lane's best member so far, its
                      * positions less one (position 256 of n = 256 fits a byte) */
    uint8_t *best;   /* [32] the block's decoding, positions ascending, less one */
    int32_t *rec;    /* [24] the block's model record */
    int32_t *anch;   /* [9] anchors during the fit */
    __device__ __forceinline__ FsSmem() {}
    __device__ __forceinline__ FsSmem(unsigned char *base)
    {
        unsigned char *p = base;
        rho = (uint32_t *)p;
        p += 258 * 4;
        msuf = (uint32_t *)p;
        p += 258 * 4;
        c0 = (uint32_t *)p;
        p += 258 * 4;
        p = (unsigned char *)(((uintptr_t)p + 15) & ~(uintptr_t)15);
        h = (T *)p;
        if (W > 1)
            p += 258 * sizeof(T);
        L = (float *)p;
        p += 256 * 4;
        pi = p;
        p += 256;
        cw = p;
        p += 256;
        stk = p;
        p += 32 * 32;
        hb = p;
        p += 32 * 32;
        best = p;
        p += 32;
        rec = (int32_t *)p;
        p += 24 * 4;
        anch = (int32_t *)p;
    }
};

template <int W>
__host__ __device__ constexpr uint32_t fs_warp_bytes()
{
    return (uint32_t)((3 * 258 * 4 + 15) / 16 * 16 + (W > 1 ? 258 * 4 * W : 0) + 256 * 4 + 256 +
                      256 + 32 * 32 + 32 * 32 + 32 + 24 * 4 + 9 * 4 + 15) /
           16 * 16;
}

/* ---------------------------------------------------------- the fit */

/* The largest chord gap over the indices of (lo, hi), the smaller index on
 * equal gaps (-1 if no gap is > 0), exactly as the one-lane loop of
 * fit_sorted finds it.  Each lane first computes its indices' gaps in
 * single precision: with M the largest |L| of the interval, a single-
 * precision gap is within 7 * 2^-24 M of the double-precision one (five
 * roundings, each of a value <= 2 M), so an index whose single-precision gap
 * is more than 2^-19 M below the largest cannot hold the largest double-
 * precision gap.  If exactly one index is left and its gap exceeds 2^-19 M,
 * its double-precision gap is positive and larger than every other one: it
 * is the answer, with no double-precision work; otherwise the remaining
 * candidates are evaluated in double precision (all of them when the curve
 * is not finite there). */
template <int W>
__device__ __forceinline__ int chord_argmax(const FsSmem<W> &sm, int lo, int hi, int lane)
{
    float M = 0.0f, g32max = 0.0f;
    for (int j = lo + lane; j <= hi; j += 32)
        M = fmaxf(M, sm.L[j - 1]);
    /* reliabilities are >= 0 (or +inf): their bit patterns order as they do */
    M = __uint_as_float(__reduce_max_sync(FULL_MASK, __float_as_uint(M)));
    const bool finite = isfinite(M);
    const float Llo = sm.L[lo - 1], rise = sm.L[hi - 1] - Llo, span = (float)(hi - lo);
    const float margin = ldexpf(M, -19);
    if (finite) {
        for (int j = lo + 1 + lane; j < hi; j += 32)
            g32max = fmaxf(g32max, fabsf(Llo + rise * (float)(j - lo) / span - sm.L[j - 1]));
        g32max = __uint_as_float(__reduce_max_sync(FULL_MASK, __float_as_uint(g32max)));
        const float cut = g32max - margin;
        uint32_t n_cand = 0;
        int cand = -1;
        for (int j = lo + 1 + lane; j < hi; j += 32)
            if (fabsf(Llo + rise * (float)(j - lo) / span - sm.L[j - 1]) >= cut) {
                n_cand++;
                cand = j;
            }
        if (__reduce_add_sync(FULL_MASK, n_cand) == 1u && g32max > margin)
            return __reduce_max_sync(FULL_MASK, (unsigned)(cand + 1)) - 1;
    }
    const float cut = g32max - margin;
    double gap = 0.0;
    int best = -1;
    for (int j = lo + 1 + lane; j < hi; j += 32) {
        if (finite && fabsf(Llo + rise * (float)(j - lo) / span - sm.L[j - 1]) < cut)
            continue;
        const double g = orbg_fit::chord_gap(sm.L, lo, hi, j);
        if (g > gap) {
            gap = g;
            best = j;
        }
    }
    /* gaps kept are >= 0 and not NaN: their bit patterns order as they do */
    unsigned long long gb = (unsigned long long)__double_as_longlong(gap);
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const unsigned long long og = __shfl_xor_sync(FULL_MASK, gb, d);
        const int oj = __shfl_xor_sync(FULL_MASK, best, d);
        if (oj >= 0 && (best < 0 || og > gb || (og == gb && oj < best))) {
            gb = og;
            best = oj;
        }
    }
    return best;
}

/* Eq. Q and Eq. quant for the anchors sm.anch[0..na-1], one segment per
 * lane: the same double operations per segment as orbg_fit::quantise, and
 * the same results (the least slope is taken over the segments in any
 * order; a NaN first slope gives the basic model as there).  Writes sm.rec,
 * which holds the basic model on entry. */
template <int W>
__device__ __forceinline__ void quantise_lanes(const FsSmem<W> &sm, int na, int divisible,
                                               int lane)
{
    using namespace orbg_fit;
    const double kFitMax = 16777216.0; /* 2^24 */
    const int m = na - 1;
    const bool mine = lane < m;
    const int a0 = sm.anch[mine ? lane : 0], a1 = sm.anch[mine ? lane + 1 : 1];
    const double sl = mine ? dvd(sub(Lj(sm.L, a1), Lj(sm.L, a0)), (double)(a1 - a0)) : 0.0;
    const double s0 = __shfl_sync(FULL_MASK, sl, 0);
    double Q = mine ? sl : s0;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1)
        Q = fmin(Q, __shfl_xor_sync(FULL_MASK, Q, d));
    if (s0 != s0)
        Q = s0; /* the first slope NaN: as the one-lane loop, no positive Q */
    if (!(Q > 0.0))
        return;
    const double rs = mine ? dvd(sl, Q) : 0.0;
    const double rl = mine ? dvd(Lj(sm.L, a0), Q) : 0.0;
    const bool bad = mine && (!(rs <= kFitMax) || !(rl <= kFitMax));
    if (__any_sync(FULL_MASK, bad))
        return;
    long long beta = 0, J = 0;
    if (mine) {
        beta = round_half_away(rs);
        J = round_half_away(rl);
    }
    const long long beta1 = __shfl_sync(FULL_MASK, beta, 0);
    if (lane == 0)
        J -= beta1;
    if (mine && divisible)
        J = round_half_away(dvd((double)J, (double)beta)) * beta;
    __syncwarp();
    if (lane == 0)
        sm.rec[0] = m;
    if (mine) {
        if (lane >= 1)
            sm.rec[lane] = a0;
        sm.rec[8 + lane] = (int32_t)J;
        sm.rec[16 + lane] = (int32_t)beta;
    }
    __syncwarp();
}

/* Sec. III-E on the ordered curve sm.L: anchors by the largest chord gap,
 * then Eq. Q / Eq. quant.  Writes sm.rec. */
template <int W>
__device__ void fit_block(const FsSmem<W> &sm, int n, int lines, int divisible, int lane)
{
    if (lane < ORBG_FIT_WORDS)
        sm.rec[lane] = 0;
    __syncwarp();
    if (lane == 0) {
        sm.rec[0] = 1;
        sm.rec[8] = 0;
        sm.rec[16] = 1;
        sm.anch[0] = 1;
        sm.anch[1] = n / 2;
    }
    __syncwarp();
    if (n < 4)
        return;
    int na = 2;
    while (na - 1 < lines) {
        const int best = chord_argmax<W>(sm, sm.anch[0], sm.anch[1], lane);
        if (best < 0)
            break;
        __syncwarp();
        if (lane == 0) {
            for (int k = na; k > 1; k--)
                sm.anch[k] = sm.anch[k - 1];
            sm.anch[1] = best;
        }
        __syncwarp();
        na++;
    }
    quantise_lanes<W>(sm, na, divisible, lane);
}

/* v of position 8 lane + 1 + i becomes the least value of that and all later
 * positions. */
__device__ __forceinline__ void suffix_minima(uint32_t (&v)[8], int lane)
{
#pragma unroll
    for (int i = 6; i >= 0; i--)
        v[i] = min(v[i], v[i + 1]);
    /* minimum over the lanes above: inclusive suffix scan, shifted by one */
    uint32_t incl = v[0];
#pragma unroll
    for (int d = 1; d < 32; d <<= 1) {
        const uint32_t o = __shfl_down_sync(FULL_MASK, incl, d);
        if (lane + d < 32)
            incl = min(incl, o);
    }
    uint32_t above = __shfl_down_sync(FULL_MASK, incl, 1);
    if (lane == 31)
        above = kRhoInf;
#pragma unroll
    for (int i = 0; i < 8; i++)
        v[i] = min(v[i], above);
}

/* rho_j from the model record (Eq. relest_seg), clamped to kRhoInf, and the
 * suffix minima.  Lane l owns positions 8l + 1 .. 8l + 8. */
template <int W>
__device__ void position_weights(const FsSmem<W> &sm, int n, int lane)
{
    const int m = sm.rec[0];
    uint32_t v[8];
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int j = 8 * lane + 1 + i;
        uint32_t r = kRhoInf;
        if (j <= n) {
            int seg = 0, Ilo = 0;
            for (int s = 1; s < m; s++)
                if (j > sm.rec[s]) {
                    seg = s;
                    Ilo = sm.rec[s];
                }
            const long long w =
                (long long)sm.rec[8 + seg] + (long long)sm.rec[16 + seg] * (long long)(j - Ilo);
            r = w < 0 ? 0u : w >= (long long)kRhoInf ? kRhoInf : (uint32_t)w;
            sm.rho[j] = r;
        }
        v[i] = r;
    }
    suffix_minima(v, lane);
#pragma unroll
    for (int i = 0; i < 8; i++) {
        const int j = 8 * lane + 1 + i;
        if (j <= n)
            sm.msuf[j] = v[i];
    }
    if (lane == 0) {
        sm.rho[n + 1] = kRhoInf;
        sm.msuf[n + 1] = kRhoInf;
    }
    __syncwarp();
}

/* ------------------------------------------------- the tree walk */

/* Is the lane's node (stack j_1..j_{t-1}, then jt) before the t-position
 * pattern other[i * ostride] in lexicographic order? */
__device__ __forceinline__ bool node_lex_less(const uint8_t *stk, int lane, int t, int jt,
                                              const uint8_t *other, int ostride)
{
    for (int i = 0; i < t; i++) {
        const int a = i < t - 1 ? (int)stk[i * 32 + lane] : jt;
        const int b = (int)other[i * ostride] + 1;
        if (a != b)
            return a < b;
    }
    return false;
}

/* Are the best members of lanes la and lb (t positions each) in
 * lexicographic order? */
__device__ __forceinline__ bool hb_lex_less(const uint8_t *hb, int la, int lb, int t)
{
    for (int i = 0; i < t; i++) {
        const int a = hb[i * 32 + la], b = hb[i * 32 + lb];
        if (a != b)
            return a < b;
    }
    return false;
}

/* Is the lane's node with the pair a < b before the t-position pattern of
 * lane `lane` of hb in lexicographic order? (t = the node's size + 2) */
__device__ __forceinline__ bool node_pair_lex_less(const uint8_t *stk, int lane, int t, int jt,
                                                   int a, int b, const uint8_t *hb)
{
    for (int i = 0; i < t; i++) {
        const int x = i < t - 3 ? (int)stk[i * 32 + lane] : i == t - 3 ? jt : i == t - 2 ? a : b;
        const int y = (int)hb[i * 32 + lane] + 1;
        if (x != y)
            return x < y;
    }
    return false;
}

/* What a pass over prefixes needs besides the node arrays: the block's pairs
 * of weights slo < s <= shi in a hash set (2^SB 32-bit slots, linear
 * probing; an entry is a 16-bit tag, the hash bits below the slot's, over
 * a - 1 and b - 1), and the least weight tb[j] that a pair of the set after
 * position j can have. */
constexpr uint32_t kFsEmpty = 0xFFFFFFFFu;
struct FsPairs {
    const uint32_t *tb;
    uint32_t *set;
};

/* multiplicative: the high bits of v times an odd constant near 2^32 /
 * golden ratio */
__device__ __forceinline__ uint32_t fs_hash(uint32_t v) { return v * 0x9E3779B1u; }

template <int SB> __device__ __forceinline__ uint32_t fs_tag(uint32_t hash)
{
    return (hash << SB) & 0xFFFF0000u;
}

/* Entry with the tag of key v, or kFsEmpty (a filter: fs_match checks). */
template <int SB> __device__ __forceinline__ uint32_t fs_find(const uint32_t *set, uint32_t v)
{
    const uint32_t x = fs_hash(v), tag = fs_tag<SB>(x);
    uint32_t slot = x >> (32 - SB);
    uint32_t e = set[slot];
    while (e != kFsEmpty && ((e ^ tag) & 0xFFFF0000u) != 0u) {
        slot = (slot + 1u) & ((1u << SB) - 1u);
        e = set[slot];
    }
    return e;
}

/* The set's pair whose whole syndrome is `full` (key v): a | b << 16, 1-based, or 0. */
template <int W, int SB>
__device__ __noinline__ uint32_t fs_match(const uint32_t *set, const uint32_t *c0,
                                          const typename Syn<W>::T *h, uint32_t v,
                                          typename Syn<W>::T full)
{
    const uint32_t x = fs_hash(v), tag = fs_tag<SB>(x);
    uint32_t slot = x >> (32 - SB);
    for (;;) {
        const uint32_t e = set[slot];
        if (e == kFsEmpty)
            return 0u;
        if (((e ^ tag) & 0xFFFF0000u) == 0u) {
            const uint32_t a = ((e >> 8) & 0xFFu) + 1u, b = (e & 0xFFu) + 1u;
            if (W == 1 ? (c0[a] ^ c0[b]) == v : sz(sx(sx(h[a], h[b]), full)))
                return a | b << 16;
        }
        slot = (slot + 1u) & ((1u << SB) - 1u);
    }
}

/* Syndrome of the lane's node on all W words. */
template <int W>
__device__ __noinline__ typename Syn<W>::T node_syndrome(const FsSmem<W> &sm, int lane, int t,
                                                         int jt, typename Syn<W>::T s0)
{
    typename Syn<W>::T P = sx(s0, sm.h[jt]);
    for (int i = 0; i < t - 1; i++)
        P = sx(P, sm.h[sm.stk[i * 32 + lane]]);
    return P;
}

/*
 * One pass over the nodes whose bound is <= Rhi.
 * MODE kFsSearch: tests every node with R <= Rhi; a lane keeps its least
 *   member (bR, bT, its positions in hb) and the bound drops to the warp's
 *   lightest member.  Returns the number of nodes tested (lane's share).
 * MODE kFsRank: counts the nodes before the block's decoding (weight Rb,
 *   Hamming weight Tb, positions sm.best): lighter, or as heavy with fewer
 *   positions, or as heavy and as many positions and lexicographically
 *   smaller.  Returns the lane's share of that count.
 * MODE kFsPairs: the nodes are prefixes (first positions) of patterns, and
 *   each is one look-up of its syndrome in the set of pairs; sm.msuf holds
 *   the least weight that a prefix position >= j and a pair after it add.
 * *guard is set (warp-uniform) if the walk exceeds `steps` iterations.
 * P, w: the walk covers class w of P (P = 1, w = 0: the whole tree): the
 * sets {j} with j = w + 1 modulo P and the larger sets whose second position
 * is w + 1 modulo P.  It walks all the depth-1 nodes, and its steps to depth
 * 2 go to the next such position ("add") or P positions on ("replace"), so
 * the big subtrees of the least reliable positions are shared out evenly.
 */
enum { kFsSearch = 0, kFsRank = 1, kFsPairs = 2 };
template <int W, int MODE, int P, int SB = 14>
__device__ uint32_t tree_pass(const FsSmem<W> &sm, int n, typename Syn<W>::T s0, int32_t Rhi,
                              int32_t Rb, int Tb, int lane, uint32_t steps, int32_t *bR,
                              int *bT, bool *guard, int w, const FsPairs *pr = nullptr)
{
    constexpr bool RANK = MODE == kFsRank, PAIRS = MODE == kFsPairs;
    const uint32_t s0w = syn_key(s0);
    bool active = false; /* an active lane's node is always untested yet */
    int t = 0, t0 = 0, jt = 0;
    uint32_t R = 0, rcur = 0, ccur = 0, syn = 0, don = 0, cnt = 0;
    /* every lane starts at once: lane l < L takes the sets whose least
     * position is l + 1 (the node {l + 1} and what its "add" branch leads to:
     * the "replace" branch at depth 1 is marked as given away), lane L the
     * sets whose least position is L + 1 or more (node {L + 1} with both
     * branches); L = min(n, 32) - 1 */
    const int last = min(n, 32) - 1;
    if (lane <= last) {
        jt = lane + 1;
        rcur = sm.rho[jt];
        ccur = sm.c0[jt];
        active = (lane < last ? rcur + (PAIRS ? pr->tb[jt] : 0u) : sm.msuf[jt]) <= (uint32_t)Rhi;
        t = 1;
        t0 = 1;
        don = lane < last ? 1u << 1 : 0u;
        R = rcur;
        syn = s0w ^ ccur;
    }
    uint32_t it = 0;
    for (;;) {
        const uint32_t act = __ballot_sync(FULL_MASK, active);
        if (act == 0)
            break;
        if (++it > steps) {
            *guard = true;
            break;
        }
        const bool tested =
            active && R + (PAIRS ? pr->tb[jt] : 0u) <= (uint32_t)Rhi &&
            (P == 1 || t != 1 || (jt - 1) % P == w);
        if (PAIRS) {
            const bool cand = tested && fs_find<SB>(pr->set, syn) != kFsEmpty;
            if (__any_sync(FULL_MASK, cand)) {
                if (cand) {
                    const uint32_t ab = fs_match<W, SB>(
                        pr->set, sm.c0, sm.h, syn,
                        W == 1 ? szero<typename Syn<W>::T>()
                               : node_syndrome<W>(sm, lane, t, jt, s0));
                    const int pa = (int)(ab & 0xFFFFu), pb = (int)(ab >> 16);
                    /* a pair not wholly after the prefix belongs to no first hit */
                    if (pa > jt) {
                        const int32_t Rp = (int32_t)(R + sm.rho[pa] + sm.rho[pb]);
                        const bool better =
                            Rp < *bR ||
                            (Rp == *bR &&
                             (t + 2 < *bT ||
                              (t + 2 == *bT && node_pair_lex_less(sm.stk, lane, t + 2, jt, pa, pb,
                                                                  sm.hb))));
                        if (better) {
                            for (int i = 0; i < t - 1; i++)
                                sm.hb[i * 32 + lane] = sm.stk[i * 32 + lane] - 1;
                            sm.hb[(t - 1) * 32 + lane] = (uint8_t)(jt - 1);
                            sm.hb[t * 32 + lane] = (uint8_t)(pa - 1);
                            sm.hb[(t + 1) * 32 + lane] = (uint8_t)(pb - 1);
                            *bR = Rp;
                            *bT = t + 2;
                        }
                    }
                }
                Rhi = min(Rhi, __reduce_min_sync(FULL_MASK, *bR));
            }
        } else if (RANK) {
            if (tested) {
                if (R < (uint32_t)Rb)
                    cnt++;
                else if (R == (uint32_t)Rb &&
                         (t < Tb || (t == Tb && node_lex_less(sm.stk, lane, t, jt, sm.best, 1))))
                    cnt++;
            }
        } else {
            cnt += tested ? 1u : 0u;
            const bool cand = tested && syn == 0u;
            if (__any_sync(FULL_MASK, cand)) {
                if (cand && (W == 1 || sz(node_syndrome<W>(sm, lane, t, jt, s0)))) {
                    const bool better =
                        (int32_t)R < *bR ||
                        ((int32_t)R == *bR &&
                         (t < *bT ||
                          (t == *bT && node_lex_less(sm.stk, lane, t, jt, sm.hb + lane, 32))));
                    if (better) {
                        for (int i = 0; i < t - 1; i++)
                            sm.hb[i * 32 + lane] = sm.stk[i * 32 + lane] - 1;
                        sm.hb[(t - 1) * 32 + lane] = (uint8_t)(jt - 1);
                        *bR = (int32_t)R;
                        *bT = t;
                    }
                }
                /* nothing heavier than the lightest member found can come first */
                Rhi = min(Rhi, __reduce_min_sync(FULL_MASK, *bR));
            }
        }
        /* the "add" child's new position: one on (at depth 1, on to the
         * warp's class) */
        const int jn = P == 1 || t != 1 ? jt + 1 : jt + 1 + ((w - jt) % P + P) % P;
        const bool okn = active && jn <= n;
        const uint32_t ms = okn ? sm.msuf[jn] : kRhoInf;
        const bool addOK = okn && R + ms <= (uint32_t)Rhi;
        /* the "replace" branch's position: one on, or P on at depth 2 */
        const int rs = t == 2 ? P : 1;
        const int jr = jt + rs;
        const bool okr = active && jr <= n;
        const uint32_t msr = P == 1 ? ms : okr ? sm.msuf[jr] : kRhoInf;
        bool replOK = okr && R - rcur + msr <= (uint32_t)Rhi && !((don >> t) & 1u);
        /* lanes without work take the replace branch of lanes about to add */
        const uint32_t idle = ~act;
        const uint32_t donors = __ballot_sync(FULL_MASK, addOK && replOK);
        bool got = false;
        if (idle != 0u && donors != 0u) {
            const uint32_t below = (1u << lane) - 1u;
            int src = lane;
            if (!active) {
                /* the r-th idle lane takes the r-th donor's branch */
                uint32_t r = __popc(idle & below);
                if (r < (uint32_t)__popc(donors)) {
                    uint32_t m = donors;
                    for (; r > 0; r--)
                        m &= m - 1u;
                    src = __ffs(m) - 1;
                }
            }
            const bool give = addOK && replOK && __popc(donors & below) < __popc(idle);
            const int st = __shfl_sync(FULL_MASK, t, src);
            const int sj = __shfl_sync(FULL_MASK, jt, src);
            const uint32_t sR = __shfl_sync(FULL_MASK, R, src);
            const uint32_t ssyn = __shfl_sync(FULL_MASK, syn, src);
            const uint32_t src_r = __shfl_sync(FULL_MASK, rcur, src);
            const uint32_t src_c = __shfl_sync(FULL_MASK, ccur, src);
            if (src != lane) {
                const int sjr = sj + (st == 2 ? P : 1); /* the donor's replace position */
                const uint32_t rn = sm.rho[sjr], cn = sm.c0[sjr];
                for (int d = 0; d < st - 1; d++)
                    sm.stk[d * 32 + lane] = sm.stk[d * 32 + src];
                t = st;
                t0 = st;
                jt = sjr;
                R = sR - src_r + rn;
                syn = ssyn ^ src_c ^ cn;
                rcur = rn;
                ccur = cn;
                don = 0;
                active = true;
                got = true;
            }
            if (give) {
                don |= 1u << t;
                replOK = false;
            }
            __syncwarp();
        }
        if (active && !got) {
            int jm = addOK ? jn : jr; /* the position the move brings in */
            bool move = addOK || replOK;
            if (addOK && t >= kDepth) {
                *guard = true; /* deeper than the stack: cannot happen within 2^26 queries */
                active = false;
                move = false;
            } else if (addOK) {
                sm.stk[(t - 1) * 32 + lane] = (uint8_t)jt;
                t++;
            } else if (replOK && (P == 1 || t != 1)) {
                /* a leaf: test up to kLeafRun of its later siblings (same
                 * prefix, last position jm = jt + 1, ...) in this step while
                 * they are leaves too; stop at one that leads further or needs
                 * the full step, and move there (or past the tested ones) */
                const uint32_t Rp = R - rcur, sp = syn ^ ccur;
                move = false;
                bool stop = false;
#pragma unroll
                for (int u = 0; u < kLeafRun; u++) {
                    if (stop)
                        break;
                    if (jm > n || Rp + sm.msuf[jm] > (uint32_t)Rhi) {
                        stop = true; /* no later sibling is reachable */
                        break;
                    }
                    const uint32_t r = sm.rho[jm], Rs = Rp + r;
                    const bool inner = jm < n && Rs + sm.msuf[jm + 1] <= (uint32_t)Rhi;
                    const bool own =
                        PAIRS ? Rs + pr->tb[jm] <= (uint32_t)Rhi &&
                                    fs_find<SB>(pr->set, sp ^ sm.c0[jm]) != kFsEmpty
                              : Rs <= (uint32_t)Rhi &&
                                    (RANK ? Rs == (uint32_t)Rb : (sp ^ sm.c0[jm]) == 0u);
                    if (inner || own) {
                        move = true;
                        stop = true;
                        break;
                    }
                    if (Rs <= (uint32_t)Rhi)
                        cnt += RANK ? (Rs < (uint32_t)Rb ? 1u : 0u) : 1u;
                    jm += rs;
                }
                if (!stop)
                    move = jm <= n && Rp + sm.msuf[jm] <= (uint32_t)Rhi;
                if (!move) {
                    /* the siblings are done: back up from the prefix */
                    R = Rp;
                    syn = sp;
                    rcur = 0u;
                    ccur = 0u;
                }
            }
            if (!move && active && !addOK) {
                /* back up until an ancestor's "replace" branch is open (it is
                 * taken at once), or the lane's part of the tree is done */
                for (;;) {
                    if (t <= t0) {
                        active = false;
                        break;
                    }
                    R -= rcur;
                    syn ^= ccur;
                    don &= ~(1u << t);
                    t--;
                    jt = sm.stk[(t - 1) * 32 + lane];
                    rcur = sm.rho[jt];
                    ccur = RANK ? 0u : sm.c0[jt];
                    jm = jt + (t == 2 ? P : 1);
                    if (jm <= n + 1 && R - rcur + sm.msuf[jm] <= (uint32_t)Rhi &&
                        !((don >> t) & 1u)) {
                        move = true;
                        break;
                    }
                }
            }
            if (move) {
                /* the rank pass needs no syndromes */
                const uint32_t rn = sm.rho[jm], cn = RANK ? 0u : sm.c0[jm];
                if (addOK) {
                    R += rn;
                    syn ^= cn;
                } else {
                    /* replace: the last position jt gives way to jm = jt + 1 */
                    R = R - rcur + rn;
                    syn ^= ccur ^ cn;
                }
                jt = jm;
                rcur = rn;
                ccur = cn;
            }
        }
    }
    *guard = __any_sync(FULL_MASK, *guard);
    return cnt;
}

/* Sum over the warp of per-lane counts below 2^32 (exact in 64 bits). */
__device__ __forceinline__ uint64_t warp_sum64(uint32_t v)
{
    const uint64_t hi = __reduce_add_sync(FULL_MASK, v >> 16);
    const uint64_t lo = __reduce_add_sync(FULL_MASK, v & 0xFFFFu);
    return (hi << 16) + lo;
}

/* ---------------------------------------------------------- one block */

/* Handover record of a block left to the search launch (ORBG_FIT_HAND_BYTES
 * bytes): its reliability order pi (n bytes), its model record (24 int32)
 * and its starting syndrome s0. */
constexpr int kHandRec = 256;
constexpr int kHandS0 = 352;
static_assert(kHandS0 + 16 <= ORBG_FIT_HAND_BYTES, "handover record too small");

/* Stage 1 of a block (the preparing launch): load, hard decision, s0; the
 * exact reliability order and the fit (steps 1-3).  A block that needs no
 * search (NaN, a hard decision that is a code word, cap 1) is finished and
 * written here; any other is appended to the open list with its handover
 * record. */
template <int K, int W>
__device__ void prepare_fitted_block(const OrbgDeviceCode &code, const float *__restrict__ llr,
                                     uint8_t *__restrict__ cw_out, uint32_t *__restrict__ q_out,
                                     uint8_t *__restrict__ ab_out, int32_t *__restrict__ rec_out,
                                     uint32_t cap, int lines, int divisible, const FsSmem<W> &sm,
                                     int lane, uint32_t b, uint32_t *__restrict__ open,
                                     unsigned long long *__restrict__ nopen,
                                     unsigned char *__restrict__ hand)
{
    typedef typename Syn<W>::T T;
    const int n = code.n;
    uint32_t key[K];
    bool nan;
    const T s0 = load_block<K, W>(code, llr, key, sm.cw, lane, &nan);
    uint32_t q = 0;
    int ab = 0;
    if (nan) {
        ab = ORBG_BLOCK_NAN;
        if (rec_out && lane < ORBG_FIT_WORDS)
            rec_out[lane] = 0;
    } else if (sz(s0) && rec_out == nullptr) {
        q = 1; /* the hard decision is a code word: query 1, whatever the model */
    } else {
#pragma unroll
        for (int k = 0; k < K; k++)
            key[k] = make_key<K>(key[k], k * 32 + lane);
        sort_block<K>(key, llr, n, lane);
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int e = lane * K + k;
            if (e < n) {
                const int idx = (int)key[k];
                sm.pi[e] = (uint8_t)idx;
                sm.L[e] = fabsf(__ldg(llr + idx));
            }
        }
        __syncwarp();
        fit_block<W>(sm, n, lines, divisible, lane);
        if (rec_out && lane < ORBG_FIT_WORDS)
            rec_out[lane] = sm.rec[lane];
        if (sz(s0)) {
            q = 1;
        } else if (cap <= 1) {
            q = cap;
            ab = ORBG_BLOCK_ABANDONED;
        } else {
            /* to the search launch */
            unsigned long long slot = 0;
            if (lane == 0)
                slot = atomicAdd(nopen, 1ull);
            slot = __shfl_sync(FULL_MASK, slot, 0);
            unsigned char *r = hand + slot * ORBG_FIT_HAND_BYTES;
            for (int e = lane; e < n; e += 32)
                r[e] = sm.pi[e];
            if (lane < ORBG_FIT_WORDS)
                reinterpret_cast<int32_t *>(r + kHandRec)[lane] = sm.rec[lane];
            if (lane == 0) {
                *reinterpret_cast<T *>(r + kHandS0) = s0;
                open[slot] = b;
            }
            __syncwarp();
            return;
        }
    }
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int i = k * 32 + lane;
        if (i < n)
            cw_out[i] = sm.cw[i];
    }
    if (lane == 0) {
        *q_out = q;
        *ab_out = (uint8_t)ab;
    }
    __syncwarp();
}
/* A block's state for the search, from its handover record and LLRs: the
 * order, the permuted columns, the hard decision and the model, then the
 * position weights.  Returns s0. */
template <int W>
__device__ typename Syn<W>::T load_record(const OrbgDeviceCode &code,
                                          const float *__restrict__ llr, const FsSmem<W> &sm,
                                          int lane, const unsigned char *__restrict__ r)
{
    typedef typename Syn<W>::T T;
    const int n = code.n;
    for (int e = lane; e < n; e += 32) {
        const int idx = (int)r[e];
        sm.pi[e] = (uint8_t)idx;
        const T col = load_col<W>(code.hcol, idx);
        sm.c0[e + 1] = syn_key(col);
        if (W > 1)
            sm.h[e + 1] = col;
        sm.cw[e] = __ldg(llr + e) > 0.0f ? 1 : 0;
    }
    if (lane == 0) {
        sm.c0[0] = 0u;
        if (W > 1)
            sm.h[0] = szero<T>();
    }
    if (lane < ORBG_FIT_WORDS)
        sm.rec[lane] = reinterpret_cast<const int32_t *>(r + kHandRec)[lane];
    __syncwarp();
    position_weights<W>(sm, n, lane);
    return *reinterpret_cast<const T *>(r + kHandS0);
}

/* Classes of the tree a CTA's warps share out, pass by pass, from a counter:
 * class k holds the sets {j} with j = k + 1 and the larger sets whose second
 * position is k + 1 modulo kClasses (many more classes than warps, so the
 * warps end a pass close together). */
constexpr int kClasses = 64; /* measured on CA-Polar[256,234]: 32 95 ms, 64 87, 128 88 */

/* Exchange area of the warps of a CTA that search one block together. */
struct FsTeam {
    unsigned int next[2];           /* the next class of a search pass, of a rank pass */
    unsigned long long c[kWarps];   /* a pass's tested nodes, per warp */
    int32_t rb[kWarps];             /* its lightest member's weight (kNoHit: none) */
    int32_t tb[kWarps];             /* that member's size */
    int32_t guard[kWarps];
    uint8_t pos[kWarps][32];        /* that member's positions */
};

/* The warp's least member of a pass (weight Rb over the warp): its size,
 * and (lanes < size) its positions in *pos_out. */
template <int W>
__device__ __forceinline__ int warp_least_member(const FsSmem<W> &sm, int lane, int32_t bR,
                                                 int bT, int32_t Rb, uint8_t *pos_out)
{
    int cl = bR == Rb ? lane : -1;
    int cT = bR == Rb ? bT : 0x7FFFFFFF;
#pragma unroll
    for (int d = 16; d >= 1; d >>= 1) {
        const int ol = __shfl_down_sync(FULL_MASK, cl, d);
        const int oT = __shfl_down_sync(FULL_MASK, cT, d);
        if (lane + d < 32 && ol >= 0 &&
            (cl < 0 || oT < cT || (oT == cT && hb_lex_less(sm.hb, ol, cl, oT)))) {
            cl = ol;
            cT = oT;
        }
    }
    cl = __shfl_sync(FULL_MASK, cl, 0);
    const int Tb = __shfl_sync(FULL_MASK, cT, 0);
    if (lane < Tb)
        pos_out[lane] = sm.hb[lane * 32 + cl];
    __syncwarp();
    return Tb;
}

/*
 * The banded search of one block (steps 5): by one warp (CTA = false), or
 * by the kWarps warps of a CTA (CTA = true), each taking classes of the
 * tree (kClasses) from a counter, each pass's counts, members and guard
 * combined through `team` (every warp takes the same decisions).
 * split > 0 (one warp): a pass without a member that tests more than
 * `split` nodes (and has not reached the cap) ends the walk with *handover
 * set, for the CTA search.  Sets *q, *ab, and *wbest (the decoding's size;
 * its positions in sm.best).
 */
template <int W, bool CTA>
__device__ void band_search(const FsSmem<W> &sm, int n, typename Syn<W>::T s0, uint32_t cap,
                            int lane, int warp, FsTeam *team, uint32_t split, uint32_t *q_out,
                            int *ab_out, int *wbest_out, bool *handover)
{
    constexpr int P = CTA ? kClasses : 1;
    uint32_t q = 0;
    int ab = 0, wbest = 0;
    *handover = false;
    /* first bound: the twelfth position's weight (about seventy patterns
     * for the basic order) */
    uint32_t r12 = lane < 12 && lane < n ? sm.rho[lane + 1] : 0u;
    r12 = __reduce_max_sync(FULL_MASK, r12);
    int32_t Rhi = (int32_t)min(max(r12, sm.msuf[1]), (uint32_t)kRmax);
    int32_t Rprev = (int32_t)sm.msuf[1] - 1;
    double Cprev = 1.0;
    const uint32_t steps = 64u * (min(cap, (uint32_t)ORBG_MAX_QUERY_CAP) + 4096u);
    for (;;) {
        int32_t bR = kNoHit;
        int bT = 0;
        bool guard = false;
        uint32_t c = 0;
        if (!CTA) {
            c = tree_pass<W, kFsSearch, 1>(sm, n, s0, Rhi, 0, 0, lane, steps, &bR, &bT, &guard, 0);
        } else {
            for (;;) {
                unsigned int k = 0;
                if (lane == 0)
                    k = atomicAdd(&team->next[0], 1u);
                k = __shfl_sync(FULL_MASK, k, 0);
                if (k >= (unsigned)kClasses)
                    break;
                const int32_t Rk = min(Rhi, __reduce_min_sync(FULL_MASK, bR));
                c += tree_pass<W, kFsSearch, P>(sm, n, s0, Rk, 0, 0, lane, steps, &bR, &bT, &guard,
                                            (int)k);
            }
        }
        uint64_t tested = warp_sum64(c);
        int32_t Rb = __reduce_min_sync(FULL_MASK, bR);
        int Tb = 0;
        if (!CTA) {
            if (Rb != kNoHit && !guard)
                Tb = warp_least_member<W>(sm, lane, bR, bT, Rb, sm.best);
        } else {
            if (Rb != kNoHit && !guard)
                Tb = warp_least_member<W>(sm, lane, bR, bT, Rb, team->pos[warp]);
            if (lane == 0) {
                team->c[warp] = tested;
                team->rb[warp] = Rb;
                team->tb[warp] = Tb;
                team->guard[warp] = guard ? 1 : 0;
            }
            __syncthreads();
            if (threadIdx.x == 0)
                team->next[0] = 0u; /* no warp takes a class again before the sync below */
            /* the team's totals and least member: weight, size, positions */
            tested = 0;
            guard = false;
            Rb = kNoHit;
            int win = -1;
            for (int v = 0; v < kWarps; v++) {
                tested += team->c[v];
                guard |= team->guard[v] != 0;
                const int32_t r = team->rb[v];
                if (r == kNoHit)
                    continue;
                bool better = win < 0 || r < Rb;
                if (!better && r == Rb) {
                    const int t = team->tb[v], tw = team->tb[win];
                    better = t < tw;
                    if (t == tw)
                        for (int i = 0; i < t; i++)
                            if (team->pos[v][i] != team->pos[win][i]) {
                                better = team->pos[v][i] < team->pos[win][i];
                                break;
                            }
                }
                if (better) {
                    win = v;
                    Rb = r;
                }
            }
            if (win >= 0) {
                Tb = team->tb[win];
                if (lane < Tb)
                    sm.best[lane] = team->pos[win][lane];
            }
            __syncthreads(); /* every warp has read the team's entries */
        }
        if (guard) {
            ab = kBlockRange;
            break;
        }
        const double C = 1.0 + (double)tested;
        if (Rb != kNoHit) {
            __syncwarp();
            uint32_t b = 0;
            if (!CTA) {
                b = tree_pass<W, kFsRank, 1>(sm, n, s0, Rb, Rb, Tb, lane, steps, &bR, &bT, &guard,
                                          0);
            } else {
                for (;;) {
                    unsigned int k = 0;
                    if (lane == 0)
                        k = atomicAdd(&team->next[1], 1u);
                    k = __shfl_sync(FULL_MASK, k, 0);
                    if (k >= (unsigned)kClasses)
                        break;
                    b += tree_pass<W, kFsRank, P>(sm, n, s0, Rb, Rb, Tb, lane, steps, &bR, &bT,
                                               &guard, (int)k);
                }
            }
            uint64_t before = warp_sum64(b);
            if (CTA) {
                if (lane == 0) {
                    team->c[warp] = before;
                    team->guard[warp] = guard ? 1 : 0;
                }
                __syncthreads();
                if (threadIdx.x == 0)
                    team->next[1] = 0u;
                before = 0;
                guard = false;
                for (int v = 0; v < kWarps; v++) {
                    before += team->c[v];
                    guard |= team->guard[v] != 0;
                }
                __syncthreads();
            }
            if (guard) {
                ab = kBlockRange;
                break;
            }
            const uint64_t rank = 2ull + before;
            if (rank <= cap) {
                q = (uint32_t)rank;
                wbest = Tb;
            } else {
                q = cap;
                ab = ORBG_BLOCK_ABANDONED;
            }
            break;
        }
        if (C >= (double)cap) {
            q = cap;
            ab = ORBG_BLOCK_ABANDONED;
            break;
        }
        if (!CTA && split > 0 && C > (double)split) {
            *handover = true;
            break;
        }
        if (Rhi >= kRmax) {
            ab = kBlockRange;
            break;
        }
        /* next bound: aim at about four times the patterns (at most a little
         * past the cap), from the growth over the last band */
        const double target = fmin(4.0 * C, 1.25 * (double)cap + 64.0);
        const double span = (double)(Rhi - Rprev);
        double delta = 2.0 * span;
        if (C > Cprev) {
            const double g = log(C / Cprev) / span;
            delta = log(target / C) / g;
        }
        delta = fmax(1.0, fmin(delta, 4.0 * span));
        Rprev = Rhi;
        Cprev = C;
        Rhi = (int32_t)fmin((double)Rhi + ceil(delta), (double)kRmax);
    }
    if (q == 0u && ab == 0)
        ab = kBlockRange;
    *q_out = q;
    *ab_out = ab;
    *wbest_out = wbest;
}

/* The outputs of a searched block: the decoding's flips on the hard
 * decision, the query count and the flag. */
template <int K, int W>
__device__ __forceinline__ void write_fitted(const FsSmem<W> &sm, int n, int lane, uint32_t q,
                                             int ab, int wbest, uint8_t *__restrict__ cw_out,
                                             uint32_t *__restrict__ q_out,
                                             uint8_t *__restrict__ ab_out)
{
    __syncwarp();
    if (lane < wbest)
        sm.cw[sm.pi[sm.best[lane]]] ^= 1;
    __syncwarp();
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int i = k * 32 + lane;
        if (i < n)
            cw_out[i] = sm.cw[i];
    }
    if (lane == 0) {
        *q_out = ab == kBlockRange ? 0u : q;
        *ab_out = (uint8_t)ab;
    }
    __syncwarp();
}

/* The scratch of one call (orbg_fitsearch_scratch_bytes): counters, the
 * open list, the lists of blocks for the two CTA searches, the handover
 * records. */
struct FsScratch {
    unsigned long long *cnt; /* [0] stage-1 queue, [1] open blocks, [2] stage-2 queue,
                              * [3] stage-4 queue, [4] blocks for stage 3, [5] stage-3 queue,
                              * [6] blocks for stage 4 */
    uint32_t *open;          /* block of each open slot */
    uint32_t *wide;          /* open slots left to stage 3 */
    uint32_t *rest;          /* open slots left to stage 4 */
    unsigned char *hand;
    __host__ __device__ FsScratch(unsigned char *base, int64_t B)
    {
        const size_t list = (4 * (size_t)B + 15) & ~(size_t)15;
        cnt = reinterpret_cast<unsigned long long *>(base);
        open = reinterpret_cast<uint32_t *>(base + 64);
        wide = reinterpret_cast<uint32_t *>(base + 64 + list);
        rest = reinterpret_cast<uint32_t *>(base + 64 + 2 * list);
        hand = base + 64 + 3 * list;
    }
};

/* Stage 1, persistent: warps take blocks from an atomic counter. */
template <int K, int W>
__global__ void __launch_bounds__(kWarps * 32, 3) orbg_fitprep_kernel(
    const __grid_constant__ OrbgDeviceCode code, const float *__restrict__ llr, int64_t B,
    uint32_t cap, int lines, int divisible, uint8_t *__restrict__ cw,
    uint32_t *__restrict__ q, uint8_t *__restrict__ ab, int32_t *__restrict__ models,
    unsigned char *__restrict__ scratch)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FsSmem<W> sm(smem + warp * fs_warp_bytes<W>());
    const FsScratch sc(scratch, B);
    const int64_t n = code.n;
    for (;;) {
        unsigned long long b = 0;
        if (lane == 0)
            b = atomicAdd(&sc.cnt[0], 1ull);
        b = __shfl_sync(FULL_MASK, b, 0);
        if (b >= (unsigned long long)B)
            break;
        prepare_fitted_block<K, W>(code, llr + (int64_t)b * n, cw + (int64_t)b * n, q + b, ab + b,
                                   models ? models + (int64_t)b * ORBG_FIT_WORDS : nullptr, cap,
                                   lines, divisible, sm, lane, (uint32_t)b, sc.open, &sc.cnt[1],
                                   sc.hand);
    }
}

/* Stage 2, persistent over the open list that stage 1 filled, one warp per
 * block; a block whose search grows past `split` nodes without
 * a member is left to stage 3. */
template <int K, int W>
__global__ void __launch_bounds__(kWarps * 32, 3) orbg_fitsearch_kernel(
    const __grid_constant__ OrbgDeviceCode code, const float *__restrict__ llr, int64_t B,
    uint32_t cap, uint32_t split, uint8_t *__restrict__ cw, uint32_t *__restrict__ q,
    uint8_t *__restrict__ ab, unsigned char *__restrict__ scratch)
{
    asm volatile("griddepcontrol.wait;" ::: "memory"); /* the launch before it is done */
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FsSmem<W> sm(smem + warp * fs_warp_bytes<W>());
    const FsScratch sc(scratch, B);
    const unsigned long long nopen = sc.cnt[1];
    const int n = code.n;
    for (;;) {
        unsigned long long i = 0;
        if (lane == 0)
            i = atomicAdd(&sc.cnt[2], 1ull);
        i = __shfl_sync(FULL_MASK, i, 0);
        if (i >= nopen)
            break;
        const int64_t b = sc.open[i];
        const auto s0 = load_record<W>(code, llr + b * n, sm, lane,
                                       sc.hand + i * ORBG_FIT_HAND_BYTES);
        uint32_t qb = 0;
        int abb = 0, wbest = 0;
        bool handover = false;
        band_search<W, false>(sm, n, s0, cap, lane, warp, nullptr, split, &qb, &abb, &wbest,
                              &handover);
        if (handover) {
            if (lane == 0)
                sc.wide[atomicAdd(&sc.cnt[4], 1ull)] = (uint32_t)i;
            __syncwarp();
            continue;
        }
        write_fitted<K, W>(sm, n, lane, qb, abb, wbest, cw + b * n, q + b, ab + b);
    }
}

/* Stage 4, persistent over the blocks stage 3 does not cover: all warps of a
 * CTA search one block's tree. */
template <int K, int W>
__global__ void __launch_bounds__(kWarps * 32, 3) orbg_fitsearch_cta_kernel(
    const __grid_constant__ OrbgDeviceCode code, const float *__restrict__ llr, int64_t B,
    uint32_t cap, uint8_t *__restrict__ cw, uint32_t *__restrict__ q,
    uint8_t *__restrict__ ab, unsigned char *__restrict__ scratch)
{
    asm volatile("griddepcontrol.wait;" ::: "memory"); /* the launch before it is done */
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ FsTeam team;
    __shared__ unsigned long long s_i;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FsSmem<W> sm(smem + warp * fs_warp_bytes<W>());
    const FsScratch sc(scratch, B);
    const unsigned long long nrest = sc.cnt[6];
    const int n = code.n;
    for (;;) {
        if (threadIdx.x == 0) {
            s_i = atomicAdd(&sc.cnt[3], 1ull);
            team.next[0] = 0u;
            team.next[1] = 0u;
        }
        __syncthreads();
        const unsigned long long k = s_i;
        __syncthreads(); /* everyone has read s_i before it changes */
        if (k >= nrest)
            break; /* uniform */
        const uint32_t i = sc.rest[k];
        const int64_t b = sc.open[i];
        const auto s0 = load_record<W>(code, llr + b * n, sm, lane,
                                       sc.hand + (size_t)i * ORBG_FIT_HAND_BYTES);
        uint32_t qb = 0;
        int abb = 0, wbest = 0;
        bool handover = false;
        band_search<W, true>(sm, n, s0, cap, lane, warp, &team, 0u, &qb, &abb, &wbest,
                             &handover);
        if (warp == 0)
            write_fitted<K, W>(sm, n, lane, qb, abb, wbest, cw + b * n, q + b, ab + b);
    }
}

/*
 * Stage 3: all warps of a CTA search one long block by pair look-ups.
 *
 * A pattern of two or more positions is a prefix and the pair a < b of its
 * last two.  The block's pairs go into a hash set of their syndromes, and a
 * walk over the prefixes alone (tree_pass, kFsPairs; about 3,600 for a
 * million patterns of a three-line model) looks up each one's syndrome,
 * which tests every pattern it starts.  Of several pairs of one syndrome the
 * set keeps the first in the order (weight, a, b): exchanging a later one in
 * a hit for it gives an earlier hit.  Orders of more than kFsChunk<K> pairs up
 * to a band's bound take the pairs in chunks of rising weight, each with its
 * own walk.
 *
 * How many patterns have weight r follows from a count over the weights:
 * counts[r] of the sets of the first j positions plus, for position j + 1,
 * counts[r - rho].  It gives the weight that holds the cap-th pattern, the
 * bands' bounds (kFsBand patterns, then sixteen times as many each) and the
 * patterns lighter than a hit.  The patterns as heavy as the hit but before
 * it are counted the same way by their number of positions, from the last
 * position to the first; in passing, for every position x that could take
 * the place of one of the hit's, the sets after x that complete it (the
 * lexicographically smaller ones).
 *
 * Blocks it does not cover (a weight of the cap-th pattern above kFsTop, a
 * hit of too many positions for the second count) go to the CTA tree search.
 * Measured on 20,000 CA-Polar[256,234] blocks of three lines at cap 5e6:
 * 51.1 ms a call when every search visited its patterns one by one (18.1 ms
 * of it in stage 2's longest warps, 35.6 in the CTAs' walks), 1.7 ms with
 * the longer searches here; 100,000 BCH(127,113) blocks 4.4 -> 1.5 ms.
 */
/* classes of the prefixes' tree (see kClasses): it is small, and each class
 * walks all its depth-1 nodes */
#ifndef ORBG_FS_CLASSES
#define ORBG_FS_CLASSES 16
#endif
constexpr int kFsClasses = ORBG_FS_CLASSES;
constexpr int kFsTop = 4095;          /* largest weight counted */
constexpr uint32_t kFsCountMax = 1u << 26; /* counts are exact below, and no cap is above */
constexpr uint32_t kFsBand = 32768;   /* patterns of the first band */
/* The set's slots for codes of K keys per lane, and how many pairs it takes
 * at once (load 0.44); the same words hold the tied-patterns count.  Half the
 * slots from n > 64 on let three CTAs share an SM instead of two (20,000
 * CA-Polar[256,234] blocks 1,430 -> 1,357 us); a short code's weights reach
 * further, and with half the count's entries a quarter of its blocks would
 * go to the tree search (80,000 RLC(64,51) blocks of four lines 709 -> 921). */
template <int K> constexpr int kFsSetBits = K >= 4 ? 13 : 14;
template <int K> constexpr uint32_t kFsChunk = 7u << (kFsSetBits<K> - 4);
template <int K> constexpr uint32_t kFsTied = 1u << kFsSetBits<K>;

/* Dynamic shared memory of the CTA. */
template <int K, int W> struct FpSmem {
    uint32_t *cum;   /* [kFsTop + 1] patterns of weight <= r */
    uint32_t *set;   /* [2^kFsSetBits<K>]; also the tied count */
    uint32_t *mpair; /* [258] least pair weight after position j */
    uint32_t *m3;    /* [258] least rho_v + mpair[v] over v >= j */
    uint32_t *mall;  /* [258] least rho over positions >= j */
    uint32_t *tb;    /* [258] a chunk's bounds: of a look-up, */
    uint32_t *lb;    /* [258] and of a subtree */
    FsSmem<W> sm;
    __device__ __forceinline__ FpSmem(unsigned char *base, int warp)
    {
        unsigned char *p = base;
        auto take = [&](size_t bytes) {
            unsigned char *r = p;
            p += (bytes + 15) & ~(size_t)15;
            return r;
        };
        set = (uint32_t *)take(4u << kFsSetBits<K>);
        cum = (uint32_t *)take(4 * (kFsTop + 1));
        sm.h = (typename Syn<W>::T *)take(W > 1 ? 258 * sizeof(typename Syn<W>::T) : 0);
        mpair = (uint32_t *)take(258 * 4);
        m3 = (uint32_t *)take(258 * 4);
        mall = (uint32_t *)take(258 * 4);
        tb = (uint32_t *)take(258 * 4);
        lb = (uint32_t *)take(258 * 4);
        sm.rho = (uint32_t *)take(258 * 4);
        sm.c0 = (uint32_t *)take(258 * 4);
        sm.rec = (int32_t *)take(24 * 4);
        sm.pi = take(256);
        sm.cw = take(256);
        sm.best = take(32);
        sm.stk = take(32 * 32 * kWarps) + 32 * 32 * warp;
        sm.hb = take(32 * 32 * kWarps) + 32 * 32 * warp;
        sm.msuf = mall; /* position_weights fills it; the walks read lb */
        sm.L = nullptr;
        sm.anch = nullptr;
    }
};
template <int K, int W> __host__ __device__ constexpr uint32_t fp_smem_bytes()
{
    return (4u << kFsSetBits<K>) + 4u * (kFsTop + 1) +
           (W > 1 ? (258u * 4u * W + 15u) / 16u * 16u : 0u) + 7u * ((258u * 4u + 15u) / 16u * 16u) +
           96u + 256u + 256u + 32u + 2u * 32u * 32u * kWarps;
}

/* cum[r] = patterns of weight <= r (the empty one included), r <= top,
 * exact below kFsCountMax, held there above; mall[j]: the least weight of
 * positions >= j.  From the last position to the first, in place: position p
 * of weight a adds the sets of later positions shifted by a, which are the
 * empty one and sets of weight mall[p + 1] or more, so that only r = a and r
 * >= a + mall[p + 1] change (a quarter of the entries where the weights rise
 * evenly). */
__device__ __forceinline__ void count_weights(const uint32_t *rho, const uint32_t *mall, int n,
                                              uint32_t top, uint32_t *cum)
{
    constexpr int kPer = (kFsTop + 32 * kWarps) / (32 * kWarps); /* entries of a thread */
    for (uint32_t r = threadIdx.x; r <= top; r += 32 * kWarps)
        cum[r] = r == 0u;
    __syncthreads();
    bool stale = false; /* thread 0 changed an entry since the last barrier */
    for (int p = n; p >= 1; p--) {
        const uint32_t a = rho[p], lo = a + mall[p + 1];
        if (a > top)
            continue;
        if (lo > top) {
            if (threadIdx.x == 0)
                cum[a]++;
            stale = true;
            continue;
        }
        if (stale)
            __syncthreads();
        stale = false;
        uint32_t v[kPer];
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            const uint32_t r = lo + threadIdx.x + (uint32_t)i * 32u * kWarps;
            if (lo + (uint32_t)i * 32u * kWarps > top)
                break;
            v[i] = r <= top ? min(cum[r] + cum[r - a], kFsCountMax) : 0u;
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < kPer; i++) {
            const uint32_t r = lo + threadIdx.x + (uint32_t)i * 32u * kWarps;
            if (lo + (uint32_t)i * 32u * kWarps > top)
                break;
            if (r <= top)
                cum[r] = v[i];
        }
        if (threadIdx.x == 0 && a < lo)
            cum[a]++;
        __syncthreads();
    }
    __syncthreads();
    if (threadIdx.x < 32u) {
        uint32_t run = 0;
        for (uint32_t base = 0; base <= top; base += 32u) {
            const uint32_t r = base + threadIdx.x;
            uint32_t v = r <= top ? cum[r] : 0u;
#pragma unroll
            for (int d = 1; d < 32; d <<= 1) {
                const uint32_t o = __shfl_up_sync(FULL_MASK, v, d);
                if ((int)threadIdx.x >= d)
                    v += o; /* at most 32 * 2^26 */
            }
            v = min(v + run, kFsCountMax);
            if (r <= top)
                cum[r] = v;
            run = __shfl_sync(FULL_MASK, v, 31);
        }
    }
    __syncthreads();
}

/* Least weight with at least `goal` patterns up to it; top + 1 if none. */
__device__ __forceinline__ uint32_t weight_holding(const uint32_t *cum, uint32_t top, uint32_t goal)
{
    uint32_t lo = 0, hi = top + 1u;
    while (lo < hi) {
        const uint32_t mid = (lo + hi) >> 1;
        if (cum[mid] >= goal)
            hi = mid;
        else
            lo = mid + 1u;
    }
    return lo;
}

/* The patterns of weight R before the T positions v (less one, ascending):
 * fewer positions, or as many and lexicographically smaller; T (R + 1) <=
 * kFsTied.  x[t (R + 1) + r] counts the sets of t positions of weight r, from
 * the last position to the first as count_weights does; t positions weigh t
 * mall[p] or more, so the rows of more positions join late.  Every thread
 * returns the count. */
__device__ __forceinline__ uint32_t count_tied(const uint32_t *rho, const uint32_t *mall, int n,
                                               uint32_t R, int T, const uint8_t *v, uint32_t *x,
                                               uint32_t *s_acc)
{
    const uint32_t row = R + 1u;
    for (uint32_t i = threadIdx.x; i < row * (uint32_t)T; i += blockDim.x)
        x[i] = i == 0u;
    if (threadIdx.x == 0)
        *s_acc = 0u;
    __syncthreads();
    /* thread 0 keeps the hit's next position below p and the weight before it */
    int k = T - 1;                 /* v[k] is the last hit position <= p */
    uint32_t head = 0;             /* weight of v[0 .. k] */
    uint32_t acc = 0;
    if (threadIdx.x == 0)
        for (int i = 0; i < T; i++)
            head += rho[v[i] + 1];
    for (int p = n; p >= 1; p--) {
        const uint32_t a = rho[p];
        if (threadIdx.x == 0) {
            if (k >= 0 && (int)v[k] + 1 == p) {
                head -= rho[p];
                k--;
            } else if (k < T - 1 && head + a <= R) {
                /* p in place of v[k + 1], any T - k - 2 positions after it */
                acc += x[(uint32_t)(T - k - 2) * row + (R - head - a)];
            }
        }
        if (a > R)
            continue;
        __syncthreads(); /* thread 0 has read its entry */
        const uint32_t least = mall[p + 1];
        /* rows of most positions first: each reads the one before it */
        for (int t = T - 1; t >= 2; t--) {
            /* may wrap where least > R, which is tested by itself (tested
             * first, in a branch of its own, it cost the kernel 1 %) */
            const uint32_t lo = a + (uint32_t)(t - 1) * least;
            if (least > R || lo > R)
                continue;
            for (uint32_t r = lo + threadIdx.x; r <= R; r += blockDim.x)
                x[(uint32_t)t * row + r] += x[(uint32_t)(t - 1) * row + (r - a)];
            __syncthreads();
        }
        if (threadIdx.x == 0 && T > 1)
            x[row + a]++; /* read by others after the barrier above, next time round */
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int t = 0; t < T; t++)
            acc += x[(uint32_t)t * row + R];
        *s_acc = acc;
    }
    __syncthreads();
    return *s_acc;
}

/* The pair (a, b) of key v into the set; the first of a syndrome in the
 * order (weight, a, b) stays. */
template <int W, int SB>
__device__ __forceinline__ void fs_insert(const FsSmem<W> &sm, uint32_t *set, int a, int b)
{
    const uint32_t v = sm.c0[a] ^ sm.c0[b];
    typename Syn<W>::T full = szero<typename Syn<W>::T>();
    if (W > 1)
        full = sx(sm.h[a], sm.h[b]);
    const uint32_t x = fs_hash(v), e = fs_tag<SB>(x) | (uint32_t)(a - 1) << 8 | (uint32_t)(b - 1);
    const uint32_t mine = (sm.rho[a] + sm.rho[b]) << 16 | (e & 0xFFFFu);
    uint32_t slot = x >> (32 - SB);
    for (;;) {
        uint32_t old = atomicCAS(set + slot, kFsEmpty, e);
        if (old == kFsEmpty)
            return;
        while (((old ^ e) & 0xFFFF0000u) == 0u) {
            const int oa = (int)((old >> 8) & 0xFFu) + 1, ob = (int)(old & 0xFFu) + 1;
            if (W == 1 ? (sm.c0[oa] ^ sm.c0[ob]) != v : !sz(sx(sx(sm.h[oa], sm.h[ob]), full)))
                break; /* another syndrome */
            if (((sm.rho[oa] + sm.rho[ob]) << 16 | (old & 0xFFFFu)) <= mine)
                return;
            const uint32_t was = atomicCAS(set + slot, old, e);
            if (was == old)
                return;
            old = was;
        }
        slot = (slot + 1u) & ((1u << SB) - 1u);
    }
}

template <int K, int W>
__global__ void __launch_bounds__(kWarps * 32, K >= 4 ? 3 : 2) orbg_fitpair_kernel(
    const __grid_constant__ OrbgDeviceCode code, const float *__restrict__ llr, int64_t B,
    uint32_t cap, uint8_t *__restrict__ cw, uint32_t *__restrict__ q,
    uint8_t *__restrict__ ab, unsigned char *__restrict__ scratch)
{
    typedef typename Syn<W>::T T;
    asm volatile("griddepcontrol.wait;" ::: "memory"); /* the launch before it is done */
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ FsTeam team;
    __shared__ unsigned long long s_i;
    __shared__ int32_t s_R;          /* lightest hit so far */
    __shared__ uint32_t s_next, s_acc;
    __shared__ int s_win, s_T;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    FpSmem<K, W> fp(smem, warp);
    const FsSmem<W> &sm = fp.sm;
    FsSmem<W> walk = fp.sm;
    walk.msuf = fp.lb;
    const FsPairs pairs{fp.tb, fp.set};
    const FsScratch sc(scratch, B);
    const unsigned long long nwide = sc.cnt[4];
    const int n = code.n;
    const uint32_t steps = 64u * (min(cap, (uint32_t)ORBG_MAX_QUERY_CAP) + 4096u);
    for (;;) {
        __syncthreads(); /* the previous block is written */
        if (threadIdx.x == 0)
            s_i = atomicAdd(&sc.cnt[5], 1ull);
        __syncthreads();
        if (s_i >= nwide)
            break; /* uniform */
        const uint32_t open = sc.wide[s_i];
        const int64_t b = sc.open[open];
        const unsigned char *rec = sc.hand + (size_t)open * ORBG_FIT_HAND_BYTES;
        for (int e = (int)threadIdx.x; e < n; e += (int)blockDim.x) {
            const int idx = (int)rec[e];
            sm.pi[e] = (uint8_t)idx;
            const T col = load_col<W>(code.hcol, idx);
            sm.c0[e + 1] = syn_key(col);
            if (W > 1)
                sm.h[e + 1] = col;
            sm.cw[e] = __ldg(llr + b * n + e) > 0.0f ? 1 : 0;
        }
        if (threadIdx.x < ORBG_FIT_WORDS)
            sm.rec[threadIdx.x] = reinterpret_cast<const int32_t *>(rec + kHandRec)[threadIdx.x];
        if (threadIdx.x == 0) {
            sm.c0[0] = 0u;
            if (W > 1)
                sm.h[0] = szero<T>();
            s_R = kNoHit;
        }
        const T s0 = *reinterpret_cast<const T *>(rec + kHandS0);
        __syncthreads();
        if (warp == 0) {
            position_weights<W>(sm, n, lane); /* rho and mall */
            uint32_t v[8];
            /* mpair[j]: the least rho_a + (least rho after a) over a > j */
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const int a = 8 * lane + 1 + i;
                v[i] = a < n ? min(sm.rho[a] + fp.mall[a + 1], kRhoInf) : kRhoInf;
            }
            suffix_minima(v, lane);
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const int a = 8 * lane + 1 + i;
                fp.mpair[a - 1] = v[i];
            }
            if (lane == 0)
                fp.mpair[256] = kRhoInf;
            __syncwarp();
#pragma unroll
            for (int i = 0; i < 8; i++) {
                const int j = 8 * lane + 1 + i;
                v[i] = j < n ? min(sm.rho[j] + fp.mpair[j], kRhoInf) : kRhoInf;
            }
            suffix_minima(v, lane);
#pragma unroll
            for (int i = 0; i < 8; i++)
                fp.m3[8 * lane + 1 + i] = v[i];
        }
        __syncthreads();
        /* single positions: thread j - 1 tests position j */
        int32_t bR = kNoHit;
        int bT = 0;
        bool guard = false;
        {
            const int j = (int)threadIdx.x + 1;
            if (j <= n && sm.rho[j] <= (uint32_t)kFsTop &&
                (W == 1 ? sm.c0[j] == syn_key(s0) : sz(sx(sm.h[j], s0)))) {
                bR = (int32_t)sm.rho[j];
                bT = 1;
                sm.hb[lane] = (uint8_t)(j - 1);
                atomicMin(&s_R, bR);
            }
        }
        __syncthreads();
        uint32_t Rb = 0, top = 0;
        bool counted = true;
        for (uint32_t goal = min(cap, kFsBand);; goal = goal > cap / 16u ? cap : goal * 16u) {
            /* the weight that holds the goal-th pattern */
            for (;;) {
                if (top != 0u) {
                    Rb = weight_holding(fp.cum, top, goal);
                    if (Rb <= top || top >= (uint32_t)kFsTop)
                        break;
                }
                top = top == 0u ? 319u : min(2u * top + 1u, (uint32_t)kFsTop);
                count_weights(sm.rho, fp.mall, n, top, fp.cum);
            }
            if (Rb > top) {
                counted = false; /* fewer patterns in all, or weights past the count */
                break;
            }
            /* chunks of pairs by weight: (slo, shi] */
            int32_t slo = -1;
            while (slo < (int32_t)Rb) {
                int32_t shi = (int32_t)Rb;
                if (n * (n - 1) / 2 > (int)kFsChunk<K>) {
                    for (uint32_t r = threadIdx.x; r <= Rb; r += blockDim.x)
                        fp.set[r] = 0u;
                    __syncthreads();
                    for (int a = 1 + warp; a < n; a += kWarps)
                        for (int c0 = a + 1; c0 <= n && sm.rho[a] + fp.mall[c0] <= Rb; c0 += 32) {
                            const int c = c0 + lane;
                            const uint32_t s = c <= n ? sm.rho[a] + sm.rho[c] : kRhoInf;
                            if ((int32_t)s > slo && s <= Rb)
                                atomicAdd(fp.set + s, 1u);
                        }
                    __syncthreads();
                    if (warp == 0) {
                        /* the largest shi with at most kFsChunk<K> pairs (a weight
                         * has far fewer) */
                        uint32_t run = 0;
                        int32_t lim = (int32_t)Rb;
                        for (uint32_t base = (uint32_t)(slo + 1); base <= Rb; base += 32u) {
                            const uint32_t r = base + (uint32_t)lane;
                            uint32_t v = r <= Rb ? fp.set[r] : 0u;
#pragma unroll
                            for (int d = 1; d < 32; d <<= 1) {
                                const uint32_t o = __shfl_up_sync(FULL_MASK, v, d);
                                if (lane >= d)
                                    v += o;
                            }
                            const uint32_t over =
                                __ballot_sync(FULL_MASK, run + v > kFsChunk<K> && r <= Rb);
                            if (over) {
                                lim = (int32_t)base + __ffs(over) - 2;
                                break;
                            }
                            run += __shfl_sync(FULL_MASK, v, 31);
                        }
                        if (lane == 0)
                            s_win = max(lim, slo + 1);
                    }
                    __syncthreads();
                    shi = s_win;
                }
                uint4 *clear = reinterpret_cast<uint4 *>(fp.set);
                for (uint32_t r = threadIdx.x; r < (1u << kFsSetBits<K>) / 4u; r += blockDim.x)
                    clear[r] = make_uint4(kFsEmpty, kFsEmpty, kFsEmpty, kFsEmpty);
                for (int j = (int)threadIdx.x; j <= n + 1; j += (int)blockDim.x) {
                    const uint32_t least = (uint32_t)(slo + 1);
                    fp.tb[j] = j <= n ? max(fp.mpair[j], least) : kRhoInf;
                    fp.lb[j] = j >= 1 && j <= n ? max(fp.m3[j], fp.mall[j] + least) : kRhoInf;
                }
                if (threadIdx.x == 0) {
                    s_next = 0u;
                }
                __syncthreads();
                for (int a = 1 + warp; a < n; a += kWarps)
                    for (int c0 = a + 1; c0 <= n && sm.rho[a] + fp.mall[c0] <= (uint32_t)shi;
                         c0 += 32) {
                        const int c = c0 + lane;
                        const int32_t s = (int32_t)(c <= n ? sm.rho[a] + sm.rho[c] : kRhoInf);
                        if (s > slo && s <= shi)
                            fs_insert<W, kFsSetBits<K>>(sm, fp.set, a, c);
                    }
                __syncthreads();
                if (threadIdx.x == 0) {
                    /* the empty prefix: a pair alone */
                    const uint32_t m = fs_match<W, kFsSetBits<K>>(fp.set, sm.c0, sm.h, syn_key(s0), s0);
                    if (m) {
                        const int pa = (int)(m & 0xFFFFu), pb = (int)(m >> 16);
                        const int32_t R = (int32_t)(sm.rho[pa] + sm.rho[pb]);
                        /* an equally heavy single position comes first */
                        if (R < bR || (R == bR && bT > 2)) {
                            bR = R;
                            bT = 2;
                            sm.hb[0] = (uint8_t)(pa - 1);
                            sm.hb[32] = (uint8_t)(pb - 1);
                            atomicMin(&s_R, R);
                        }
                    }
                }
                __syncwarp();
                for (;;) {
                    unsigned int k = 0;
                    if (lane == 0)
                        k = atomicAdd(&s_next, 1u);
                    k = __shfl_sync(FULL_MASK, k, 0);
                    if (k >= (unsigned)kFsClasses)
                        break;
                    const int32_t Rk = min((int32_t)Rb, *((volatile int32_t *)&s_R));
                    const int32_t was = __reduce_min_sync(FULL_MASK, bR);
                    tree_pass<W, kFsPairs, kFsClasses, kFsSetBits<K>>(walk, n, s0, Rk, 0, 0, lane, steps, &bR, &bT,
                                                     &guard, (int)k, &pairs);
                    const int32_t now = __reduce_min_sync(FULL_MASK, bR);
                    if (lane == 0 && now < was)
                        atomicMin(&s_R, now);
                }
                __syncthreads();
                slo = shi;
                if (s_R <= (int32_t)Rb && slo + 1 > s_R)
                    break; /* later pairs are heavier than the hit (uniform) */
            }
            if (s_R <= (int32_t)Rb || goal >= cap)
                break;
        }
        if (!counted) {
            __syncthreads(); /* everyone has left the search before s_R changes */
            if (threadIdx.x == 0)
                sc.rest[atomicAdd(&sc.cnt[6], 1ull)] = open;
            continue;
        }
        const int32_t R = s_R;
        const bool hit = R <= (int32_t)Rb;
        /* the team's first member of that weight */
        if (lane == 0) {
            team.rb[warp] = kNoHit;
            team.guard[warp] = guard ? 1 : 0;
        }
        __syncwarp();
        if (hit && __any_sync(FULL_MASK, bR == R)) {
            const int Tw = warp_least_member<W>(sm, lane, bR, bT, R, team.pos[warp]);
            if (lane == 0) {
                team.rb[warp] = R;
                team.tb[warp] = Tw;
            }
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            int win = -1;
            bool bad = false;
            for (int v = 0; v < kWarps; v++) {
                bad |= team.guard[v] != 0;
                if (team.rb[v] == kNoHit)
                    continue;
                bool better = win < 0 || team.tb[v] < team.tb[win];
                if (!better && team.tb[v] == team.tb[win])
                    for (int i = 0; i < team.tb[v]; i++)
                        if (team.pos[v][i] != team.pos[win][i]) {
                            better = team.pos[v][i] < team.pos[win][i];
                            break;
                        }
                if (better)
                    win = v;
            }
            s_win = bad ? -2 : win;
            s_T = win >= 0 ? team.tb[win] : 0;
        }
        __syncthreads();
        const int win = s_win, Tb = s_T;
        if (win == -2 || (hit && (uint32_t)Tb * ((uint32_t)R + 1u) > kFsTied<K>)) {
            if (threadIdx.x == 0)
                sc.rest[atomicAdd(&sc.cnt[6], 1ull)] = open;
            continue;
        }
        uint32_t rank = 0xFFFFFFFFu;
        if (hit) {
            rank = 1u + (R > 0 ? fp.cum[R - 1] : 0u) +
                   count_tied(sm.rho, fp.mall, n, (uint32_t)R, Tb, team.pos[win], fp.set, &s_acc);
            if (warp == 0 && lane < Tb)
                sm.best[lane] = team.pos[win][lane];
        }
        const bool ok = rank <= cap;
        if (warp == 0)
            write_fitted<K, W>(sm, n, lane, ok ? rank : cap, ok ? 0 : ORBG_BLOCK_ABANDONED,
                               ok ? Tb : 0, cw + b * n, q + b, ab + b);
    }
}

template <int K, int W>
int launch_fitsearch(const OrbgDeviceCode &code, const float *llr, int64_t B, uint32_t cap,
                     int lines, int divisible, uint8_t *cw, uint32_t *q, uint8_t *ab,
                     int32_t *models, unsigned char *scratch, void *stream)
{
    auto k1 = orbg_fitprep_kernel<K, W>;
    auto k2 = orbg_fitsearch_kernel<K, W>;
    auto k3 = orbg_fitpair_kernel<K, W>;
    auto k4 = orbg_fitsearch_cta_kernel<K, W>;
    const size_t smem = (size_t)fs_warp_bytes<W>() * kWarps;
    int g1 = 0, g2 = 0, g3 = 0, g4 = 0;
    int rc = orbg_grid_for((const void *)k1, kWarps * 32, smem, 0, &g1);
    if (rc == 0)
        rc = orbg_grid_for((const void *)k2, kWarps * 32, smem, 0, &g2);
    if (rc == 0)
        rc = orbg_grid_for((const void *)k3, kWarps * 32, fp_smem_bytes<K, W>(), 0, &g3);
    if (rc == 0)
        rc = orbg_grid_for((const void *)k4, kWarps * 32, smem, 0, &g4);
    if (rc != 0)
        return rc;
    const bool few = B * code.n <= kFewPositions && (code.r <= 14 || B <= kFewBlocks);
    const uint32_t most = few                                   ? kSplitFew
                          : B <= 2 * (int64_t)g2 * kWarps ? kSplitSmall
                                                          : kSplit;
    const uint32_t split = most < cap / 4u ? most : cap / 4u;
    const int64_t need = (B + kWarps - 1) / kWarps;
    if (g1 > need)
        g1 = (int)need;
    if (g2 > need)
        g2 = (int)need;
    if (g3 > B)
        g3 = (int)B;
    if (g4 > B)
        g4 = (int)B;
    cudaStream_t st = (cudaStream_t)stream;
    cudaError_t e = cudaMemsetAsync(scratch, 0, 64, st);
    if (e != cudaSuccess)
        return (int)e;
    k1<<<g1, kWarps * 32, smem, st>>>(code, llr, B, cap, lines, divisible, cw, q, ab, models,
                                      scratch);
    if ((e = cudaGetLastError()) != cudaSuccess)
        return (int)e;
    /* the further launches come on while the one before ends (each waits for
     * it first): four in a row cost a batch of ten blocks 3 us more than three */
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.blockDim = dim3(kWarps * 32);
    cfg.stream = st;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    cfg.gridDim = dim3((unsigned)g2);
    cfg.dynamicSmemBytes = smem;
    if ((e = cudaLaunchKernelEx(&cfg, k2, code, llr, B, cap, split, cw, q, ab, scratch)) !=
        cudaSuccess)
        return (int)e;
    cfg.gridDim = dim3((unsigned)g3);
    cfg.dynamicSmemBytes = fp_smem_bytes<K, W>();
    if ((e = cudaLaunchKernelEx(&cfg, k3, code, llr, B, cap, cw, q, ab, scratch)) != cudaSuccess)
        return (int)e;
    cfg.gridDim = dim3((unsigned)g4);
    cfg.dynamicSmemBytes = smem;
    return (int)cudaLaunchKernelEx(&cfg, k4, code, llr, B, cap, cw, q, ab, scratch);
}

}  // namespace orbg_fitsearch
