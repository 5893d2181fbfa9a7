/*
 * orbg_decode_block.cuh -- per-block device code of the basic-ORBGRAND
 * decoder, shared by the plain and the batched kernels.
 *
 * Decoding one received block (Algorithm 1 with the basic ORBGRAND
 * generator, Sec. III-B):
 *   1. coalesced load of the n FP32 LLRs; hard decision y_i = [L_i > 0];
 *      reliability key (FP32 bits of |L_i|, i) (Sec. III-A); starting
 *      syndrome s0 = H y (Sec. I).  If s0 = 0, y is a codeword and query 1
 *      (the zero pattern) decodes: no sort is needed;
 *   2. the reliability order pi (Sec. III-A): its leading ranks, as many as
 *      the stage of the search uses, extracted as warp minima; only an order
 *      that uses more than 128 of them takes a warp bitonic sort of the keys
 *      (the paper names bitonic sorting networks as one option, Sec. IV-B);
 *   3. permuted columns hperm[p] = H[:, pi_p] into shared memory, after a
 *      zero column read by unused prefix slots;
 *   4. past the flat table, every pattern of weight >= 2 is a prefix and a
 *      pair of its last two positions: the block's pairs go into a filter
 *      of their syndromes (and, in a CTA, a hash set behind it), and each
 *      prefix is one look-up of s0 (+) prefix
 *      (orbg_internal.h says why the first pair of a syndrome is enough, how
 *      a hit's query index is formed and when no later prefix can beat it);
 *   5. codeword y (+) z* (or y if abandoned), query count, abandon flag.
 *
 * Two ways to run step 4: one warp takes its block through the first bands
 * of the order (decode_block_warp), with a small table of its own; all warps
 * of a CTA share one block and its whole set of pairs (decode_block_cta).
 * Every loop is bounded by the tables' sizes or the hash sets'; no thread
 * waits on another's progress beyond __syncthreads.
 */
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "orbg_internal.h"

#define FULL_MASK 0xFFFFFFFFu
#define ORBG_NONE 0xFFFFFFFFu

namespace orbg_dev {

/* ---------------------------------------------------------------- vectors */

template <int W> struct Syn;
template <> struct Syn<1> { typedef uint32_t T; };
template <> struct Syn<2> { typedef uint2 T; };
template <> struct Syn<4> { typedef uint4 T; };

__device__ __forceinline__ uint32_t sx(uint32_t a, uint32_t b) { return a ^ b; }
__device__ __forceinline__ uint2 sx(uint2 a, uint2 b) { return make_uint2(a.x ^ b.x, a.y ^ b.y); }
__device__ __forceinline__ uint4 sx(uint4 a, uint4 b)
{
    return make_uint4(a.x ^ b.x, a.y ^ b.y, a.z ^ b.z, a.w ^ b.w);
}
__device__ __forceinline__ bool sz(uint32_t a) { return a == 0u; }
__device__ __forceinline__ bool sz(uint2 a) { return (a.x | a.y) == 0u; }
__device__ __forceinline__ bool sz(uint4 a) { return (a.x | a.y | a.z | a.w) == 0u; }
template <typename T> __device__ __forceinline__ T szero();
template <> __device__ __forceinline__ uint32_t szero<uint32_t>() { return 0u; }
template <> __device__ __forceinline__ uint2 szero<uint2>() { return make_uint2(0u, 0u); }
template <> __device__ __forceinline__ uint4 szero<uint4>() { return make_uint4(0u, 0u, 0u, 0u); }

template <int W>
__device__ __forceinline__ typename Syn<W>::T load_col(const uint32_t *__restrict__ hcol, int j)
{
    typedef typename Syn<W>::T T;
    return __ldg(reinterpret_cast<const T *>(hcol) + j);
}

__device__ __forceinline__ uint64_t shfl_xor_u64(uint64_t v, int m)
{
    uint32_t lo = __shfl_xor_sync(FULL_MASK, (uint32_t)v, m);
    uint32_t hi = __shfl_xor_sync(FULL_MASK, (uint32_t)(v >> 32), m);
    return ((uint64_t)hi << 32) | lo;
}

/* Shared memory of one block in flight: hperm[n+1] full syndromes, then
 * (for W > 1) h0[n+1], the key of each, then pi[256].  Entry 0 of hperm and
 * h0 is a zero column (BlockSmem). */
__host__ __device__ __forceinline__ uint32_t block_smem_bytes(int n, int w32)
{
    uint32_t h = (uint32_t)(n + 1) * 4u * (uint32_t)w32;
    h = (h + 15u) & ~15u;
    uint32_t h0 = w32 > 1 ? (((uint32_t)(n + 1) * 4u + 15u) & ~15u) : 0u;
    return h + h0 + 256u;
}

/* h[r] (and h0[r]) is the column of sorted position r, 0 <= r < n; the
 * entry before it, h[-1], is the zero column, so a 1-based position p (0 =
 * none) reads h[p - 1] with no test. */
template <int W> struct BlockSmem {
    typedef typename Syn<W>::T T;
    T *h;
    uint32_t *h0;
    uint8_t *pi;
    __device__ __forceinline__ BlockSmem(unsigned char *base, int n)
    {
        h = reinterpret_cast<T *>(base) + 1;
        unsigned char *p = base + (((uint32_t)(n + 1) * sizeof(T) + 15u) & ~15u);
        if (W > 1) {
            h0 = reinterpret_cast<uint32_t *>(p) + 1;
            p += ((uint32_t)(n + 1) * 4u + 15u) & ~15u;
        } else {
            h0 = reinterpret_cast<uint32_t *>(base) + 1;
        }
        pi = p;
    }
};

/* A 32-bit key of a syndrome, linear over GF(2) so that the key of a sum is
 * the XOR of the keys; the syndrome itself up to 32 bits.  Longer ones add
 * the further words through an invertible linear mix (xorshift steps, after
 * Marsaglia): with the first word alone, the unit columns of a systematic H
 * beyond row 32 would all have key 0 and share their sums' keys. */
__device__ __forceinline__ uint32_t key_mix(uint32_t v)
{
    v ^= v << 13;
    v ^= v >> 17;
    return v ^ (v << 5);
}
__device__ __forceinline__ uint32_t syn_key(uint32_t v) { return v; }
__device__ __forceinline__ uint32_t syn_key(uint2 v) { return v.x ^ key_mix(v.y); }
__device__ __forceinline__ uint32_t syn_key(uint4 v)
{
    return v.x ^ key_mix(v.y ^ key_mix(v.z ^ key_mix(v.w)));
}

/* LLR reads: from shared memory (LS, staged ahead by the batched kernel)
 * or from global memory through the read-only path. */
template <bool LS>
__device__ __forceinline__ float llr_at(const float *__restrict__ llr, int i)
{
    if (LS)
        return llr[i];
    return __ldg(llr + i);
}

/* Sort keys are 32 bits: (|L| bits with the low DROP bits dropped) << IB | i,
 * with IB index bits (32 K <= 2^IB).  The truncation merges reliabilities
 * that differ only in the dropped bits; inside such a tie the key orders by
 * index, which is the exact order unless the full bits disagree -- checked
 * after the sort (sort_block). */
template <int K> struct KeyBits {
    static constexpr int IB = K == 1 ? 5 : K == 2 ? 6 : K == 4 ? 7 : 8; /* 32*K <= 2^IB */
    static constexpr int DROP = IB - 1;                                  /* 31 + IB - DROP = 32 */
    static constexpr uint32_t IMASK = (1u << IB) - 1u;
};

/* ------------------------------------------------------- step 1: load */

/* A sort key of received position i from the bits of |L_i|. */
template <int K> __device__ __forceinline__ uint32_t make_key(uint32_t bits, int i)
{
    typedef KeyBits<K> KB;
    return ((bits >> KB::DROP) << KB::IB) | ((uint32_t)i & KB::IMASK);
}

/* Loads the block: the hard decision y into cw (if not NULL), the bits of
 * |L| of the lane's K positions (all ones past n) into bits[], and returns
 * s0 = H y, identical in every lane.  *nan is warp-uniform.  The warp's
 * ballots of L > 0 are y; lane i holds row i of H (and rows 32 + i, ... of
 * longer syndromes), and the parity of its AND with y is bit i of s0: the
 * row loads do not wait for the LLRs, and nothing is summed over lanes. */
template <int K, int W, bool LS = false>
__device__ __forceinline__ typename Syn<W>::T load_block(const OrbgDeviceCode &code,
                                                         const float *__restrict__ llr,
                                                         uint32_t (&bits)[K], uint8_t *cw,
                                                         int lane, bool *nan_out)
{
    const int n = code.n;
    uint32_t row[W][K], y[K];
#pragma unroll
    for (int w = 0; w < W; w++)
#pragma unroll
        for (int k = 0; k < K; k++)
            row[w][k] = __ldg(code.hrow + (w * K + k) * 32 + lane);
    bool nan = false;
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int i = k * 32 + lane;
        const bool in = i < n;
        const float L = in ? llr_at<LS>(llr, i) : 0.0f;
        const uint32_t a = __float_as_uint(L) & 0x7FFFFFFFu;
        nan |= a > 0x7F800000u;
        y[k] = __ballot_sync(FULL_MASK, L > 0.0f);
        if (in && cw != nullptr)
            cw[i] = L > 0.0f ? 1 : 0;
        bits[k] = in ? a : 0xFFFFFFFFu;
    }
    uint32_t s[W];
#pragma unroll
    for (int w = 0; w < W; w++) {
        uint32_t acc = 0;
#pragma unroll
        for (int k = 0; k < K; k++)
            acc ^= row[w][k] & y[k];
        s[w] = __ballot_sync(FULL_MASK, (__popc(acc) & 1) != 0);
    }
    *nan_out = __any_sync(FULL_MASK, nan);
    typename Syn<W>::T s0;
    if constexpr (W == 1)
        s0 = s[0];
    else if constexpr (W == 2)
        s0 = make_uint2(s[0], s[1]);
    else
        s0 = make_uint4(s[0], s[1], s[2], s[3]);
    return s0;
}

/* ------------------------------------------------------- step 2: sort */

/* Bitonic sort of 32*K unique keys held K per lane; afterwards position
 * e = lane*K + k holds the e-th smallest.  The network's merge levels and
 * its strides across lanes are loops (the compare-exchanges of one step,
 * over the lane's K keys, are unrolled): the code stays small enough to
 * remain in the instruction cache while the warps of an SM sort block after
 * block, where the fully unrolled network (about 1,300 instructions for
 * K = 8) was fetched anew for every block; the fully unrolled one also cost
 * a single code's kernel 1 to 4 % once phase 1 sorts few blocks in full). */
template <int K>
__device__ __forceinline__ void sort_keys(uint64_t (&key)[K], int lane)
{
#pragma unroll 1
    for (int size = 2; size <= 32 * K; size <<= 1) {
#pragma unroll 1
        for (int stride = size >> 1; stride >= K; stride >>= 1) {
            const int lm = stride / K;
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int e = lane * K + k;
                uint64_t o = shfl_xor_u64(key[k], lm);
                bool asc = (e & size) == 0;
                bool lower = (e & stride) == 0;
                uint64_t mn = key[k] < o ? key[k] : o;
                uint64_t mx = key[k] < o ? o : key[k];
                key[k] = (lower == asc) ? mn : mx;
            }
        }
#pragma unroll
        for (int stride = K / 2; stride > 0; stride >>= 1) {
            if (stride > (size >> 1))
                continue;
#pragma unroll
            for (int k = 0; k < K; k++) {
                if ((k & stride) == 0) {
                    const int k2 = k | stride;
                    const int e = lane * K + k;
                    bool asc = (e & size) == 0;
                    uint64_t a = key[k], b = key[k2];
                    bool sw = asc ? (a > b) : (a < b);
                    key[k] = sw ? b : a;
                    key[k2] = sw ? a : b;
                }
            }
        }
    }
}

/* Bitonic sort of 32*K unique 32-bit keys held K per lane (loops as
 * sort_keys). */
template <int K>
__device__ __forceinline__ void bitonic32(uint32_t (&key)[K], int lane)
{
#pragma unroll 1
    for (int size = 2; size <= 32 * K; size <<= 1) {
#pragma unroll 1
        for (int stride = size >> 1; stride >= K; stride >>= 1) {
            const int lm = stride / K;
#pragma unroll
            for (int k = 0; k < K; k++) {
                const int e = lane * K + k;
                const uint32_t o = __shfl_xor_sync(FULL_MASK, key[k], lm);
                const bool takemin = ((e & size) == 0) == ((e & stride) == 0);
                key[k] = takemin ? min(key[k], o) : max(key[k], o);
            }
        }
#pragma unroll
        for (int stride = K / 2; stride > 0; stride >>= 1) {
            if (stride > (size >> 1))
                continue;
#pragma unroll
            for (int k = 0; k < K; k++) {
                if ((k & stride) == 0) {
                    const int k2 = k | stride;
                    const int e = lane * K + k;
                    const bool asc = (e & size) == 0;
                    const uint32_t lo = min(key[k], key[k2]), hi = max(key[k], key[k2]);
                    key[k] = asc ? lo : hi;
                    key[k2] = asc ? hi : lo;
                }
            }
        }
    }
}

/*
 * Sort the 32-bit keys, then check every adjacent pair whose truncated
 * reliabilities are equal against the full bits; if any is out of order,
 * sort exact 64-bit keys (bits << 32 | i) rebuilt from the LLRs instead.
 * Afterwards key[k] holds the received index of sorted position lane*K + k.
 */
template <int K, bool LS = false>
__device__ __forceinline__ void sort_block(uint32_t (&key)[K], const float *__restrict__ llr,
                                           int n, int lane)
{
    typedef KeyBits<K> KB;
    bitonic32<K>(key, lane);
    bool bad = false;
    const uint32_t next_first = __shfl_down_sync(FULL_MASK, key[0], 1);
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int e = lane * K + k;
        const uint32_t nxt = (k + 1 < K) ? key[k + 1 < K ? k + 1 : k] : next_first;
        if (e + 1 < n && (key[k] >> KB::IB) == (nxt >> KB::IB)) {
            const uint32_t ba =
                __float_as_uint(llr_at<LS>(llr, (int)(key[k] & KB::IMASK))) & 0x7FFFFFFFu;
            const uint32_t bb =
                __float_as_uint(llr_at<LS>(llr, (int)(nxt & KB::IMASK))) & 0x7FFFFFFFu;
            bad |= ba > bb;
        }
    }
    if (__any_sync(FULL_MASK, bad)) {
        uint64_t k64[K];
#pragma unroll
        for (int k = 0; k < K; k++) {
            const int i = k * 32 + lane;
            const uint32_t bits =
                i < n ? (__float_as_uint(llr_at<LS>(llr, i)) & 0x7FFFFFFFu) : 0xFFFFFFFFu;
            k64[k] = ((uint64_t)bits << 32) | (uint32_t)i;
        }
        sort_keys<K>(k64, lane);
#pragma unroll
        for (int k = 0; k < K; k++)
            key[k] = (uint32_t)k64[k];
        return;
    }
#pragma unroll
    for (int k = 0; k < K; k++)
        key[k] &= KB::IMASK;
}

/* ------------------------------------------------- step 3: permutation */

template <int K, int W>
__device__ __forceinline__ void build_perm(const OrbgDeviceCode &code, const uint32_t (&key)[K],
                                           const BlockSmem<W> &sm, int lane)
{
    const int n = code.n;
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int e = lane * K + k;
        if (e < n) {
            const int idx = (int)key[k];
            sm.pi[e] = (uint8_t)idx;
            const typename Syn<W>::T col = load_col<W>(code.hcol, idx);
            sm.h[e] = col;
            if (W > 1)
                sm.h0[e] = syn_key(col);
        }
    }
    if (lane == 0) {
        sm.h[-1] = szero<typename Syn<W>::T>();
        if (W > 1)
            sm.h0[-1] = 0u;
    }
}

/* ------------------------------------- step 2': the leading ranks only */

/*
 * Each stage of the search (a flat step, a band, the handover to a CTA)
 * reaches only so many of the least reliable positions.  Instead of a full
 * sort the smallest keys are extracted one at a time, a warp minimum per
 * rank, until the ranks the stage needs are known.  Each lane first sorts
 * its own K keys, so its smallest is key[0].
 */
template <int K>
__device__ __forceinline__ void sort_lane(uint32_t (&key)[K])
{
#pragma unroll
    for (int i = 0; i < K; i++)
#pragma unroll
        for (int j = 0; j + 1 < K - i; j++) {
            const uint32_t lo = min(key[j], key[j + 1]), hi = max(key[j], key[j + 1]);
            key[j] = lo;
            key[j + 1] = hi;
        }
}

/* Ranks taken one at a time at most; beyond, a full sort is cheaper.  A
 * handover to phase 2 at cap 1e6 needs 82: sorted in full, 256 keys cost
 * phase 1 a bitonic network and, in one block of three, a second one on exact
 * keys for a tie somewhere among them. */
constexpr int kMostRanks = 128;

/* The lane's keys, ascending: its smallest, and how the next ones follow.
 * Up to four keys shift down in registers; eight (n > 128) go to a list in
 * shared memory, where taking one costs a load instead of eight moves and
 * the registers are free for the search (about 20 warp instructions a rank
 * in registers, 13 with the list).  The list ends on a key past all. */
template <int K> constexpr bool kKeyList = K >= 8;
template <int K> __host__ __device__ constexpr uint32_t key_list_bytes() { return kKeyList<K> ? (K + 1) * 128u : 0u; }
template <int K> struct LaneKeys {
    uint32_t key[K];
    __device__ __forceinline__ LaneKeys(const uint32_t (&sorted)[K], uint32_t *, int)
    {
#pragma unroll
        for (int k = 0; k < K; k++)
            key[k] = sorted[k];
    }
    __device__ __forceinline__ uint32_t first() const { return key[0]; }
    __device__ __forceinline__ void take(bool mine)
    {
        if (mine) {
#pragma unroll
            for (int k = 0; k + 1 < K; k++)
                key[k] = key[k + 1];
            key[K - 1] = 0xFFFFFFFFu;
        }
    }
};
template <> struct LaneKeys<8> {
    uint32_t cur;
    const uint32_t *at;
    __device__ __forceinline__ LaneKeys(const uint32_t (&sorted)[8], uint32_t *list, int lane)
    {
#pragma unroll
        for (int k = 1; k < 8; k++)
            list[k * 32 + lane] = sorted[k];
        list[8 * 32 + lane] = 0xFFFFFFFFu;
        cur = sorted[0];
        at = list + 32 + lane;
    }
    __device__ __forceinline__ uint32_t first() const { return cur; }
    __device__ __forceinline__ void take(bool mine)
    {
        if (mine) {
            cur = *at;
            at += 32;
        }
    }
};

/* Extracts ranks have .. upto-1: pi[r] is rank r's received index.  Returns
 * true if two consecutive ranks (this call's or the last earlier one, in
 * *prev) have equal truncated reliabilities: then the truncated order may
 * differ from the exact one and the caller sorts exactly instead. */
template <int K>
__device__ __forceinline__ bool extract_ranks(LaneKeys<K> &keys, int have, int upto,
                                              uint32_t *prev, uint8_t *pi)
{
    typedef KeyBits<K> KB;
    bool tie = false;
    uint32_t pv = *prev;
    for (int r = have; r < upto; r++) {
        const uint32_t g = __reduce_min_sync(FULL_MASK, keys.first());
        tie |= (g >> KB::IB) == (pv >> KB::IB);
        const bool mine = keys.first() == g;
        if (mine)
            pi[r] = (uint8_t)(g & KB::IMASK);
        keys.take(mine);
        pv = g;
    }
    *prev = pv;
    return tie;
}

/* Permuted columns of ranks lo .. hi-1, whose received indices are in pi. */
template <int W>
__device__ __forceinline__ void perm_ranks(const OrbgDeviceCode &code, int lo, int hi,
                                           const BlockSmem<W> &sm, int lane)
{
    for (int r = lo + lane; r < hi; r += 32) {
        const typename Syn<W>::T col = load_col<W>(code.hcol, (int)sm.pi[r]);
        sm.h[r] = col;
        if (W > 1)
            sm.h0[r] = syn_key(col);
    }
}

/* The K truncated keys of a lane, in load order. */
template <int K, bool LS>
__device__ __forceinline__ void make_keys(const float *__restrict__ llr, int n, int lane,
                                          uint32_t (&key)[K])
{
#pragma unroll
    for (int k = 0; k < K; k++) {
        const int i = k * 32 + lane;
        const uint32_t bits =
            i < n ? (__float_as_uint(llr_at<LS>(llr, i)) & 0x7FFFFFFFu) : 0xFFFFFFFFu;
        key[k] = make_key<K>(bits, i);
    }
}

/* ------------------------------------------- step 4: pair look-ups */

/*
 * The pairs of a block are looked up through a filter: 2^bits bits, of which
 * each pair sets two.  A look-up reads two words and needs no loop: with a
 * hash set alone a warp step waited for its longest probe sequence (80 warp
 * instructions a step of 32 look-ups, 45 with the filter).  Both hashes are
 * multiplicative (the high bits of the key times an odd constant, the first
 * near 2^32 / golden ratio, the second the first multiplier of MurmurHash3's
 * final mix, A. Appleby): the low bits of one product would repeat where the
 * code's columns differ in few rows.
 */
__device__ __forceinline__ uint32_t pair_hash(uint32_t v) { return v * 0x9E3779B1u; }
__device__ __forceinline__ void filter_add(uint32_t *filter, uint32_t bits, uint32_t v)
{
    const uint32_t i = pair_hash(v) >> (32u - bits), j = (v * 0x85EBCA6Bu) >> (32u - bits);
    atomicOr(filter + (i >> 5), 1u << (i & 31u));
    atomicOr(filter + (j >> 5), 1u << (j & 31u));
}
/* May the filter hold a pair of key v? */
__device__ __forceinline__ bool filter_has(const uint32_t *filter, uint32_t bits, uint32_t v)
{
    const uint32_t i = pair_hash(v) >> (32u - bits), j = (v * 0x85EBCA6Bu) >> (32u - bits);
    return ((filter[i >> 5] >> (i & 31u)) & (filter[j >> 5] >> (j & 31u)) & 1u) != 0u;
}

/* A warp's own: 2^14 bits for the 484 pairs of the second band, so that 0.3 %
 * of look-ups pass by chance, and the pairs' keys in order, which the warp
 * looks through for a key that passed. */
constexpr uint32_t kWarpFilterBits = 14;
constexpr uint32_t kWarpFilterBytes = (1u << kWarpFilterBits) / 8u;
constexpr uint32_t kWarpPairBytes = kWarpFilterBytes + ((ORBG_BAND2_PAIRS * 4u + 15u) & ~15u);

/* A CTA's for `npairs` pairs at once, at most kPairChunk: at least 64 bits a pair (2^17 for the 1,640 of cap 1e6), and a
 * hash set behind it of at least two slots a pair, linear probing, in which
 * every lane finds its own pair (codes of few parity bits hit often).  An
 * entry is the pair's index in the chunk (low 12 bits) under the hash bits
 * below the slot's; of pairs of equal syndrome the first stays. */
constexpr uint32_t kIdMask = 0xFFFu;
constexpr uint32_t kPairChunk = ORBG_PAIR_CHUNK; /* 4095: entry kEmpty is never a pair's */
constexpr uint32_t kEmpty = 0xFFFFFFFFu;
__host__ __device__ __forceinline__ uint32_t pair_filter_bits(uint32_t npairs)
{
    uint32_t b = 12;
    while (b < 18 && (1u << b) < 64u * npairs)
        b++;
    return b;
}
__host__ __device__ __forceinline__ uint32_t pair_slot_bits(uint32_t npairs)
{
    return pair_filter_bits(npairs) - 5u;
}
/* Keys of the subsets of the eight lightest positions, then of the next
 * eight: a prefix record names its light positions by two bytes. */
constexpr uint32_t kMaskBytes = 512 * 4;
__host__ __device__ __forceinline__ uint32_t pair_smem_bytes(uint32_t npairs)
{
    return kMaskBytes + (1u << pair_filter_bits(npairs)) / 8u + (4u << pair_slot_bits(npairs));
}
__device__ __forceinline__ uint32_t slot_tag(uint32_t hash, uint32_t bits)
{
    return (hash << bits) & ~kIdMask;
}

/* Pair id (of the chunk from lo) into the CTA's filter and set. */
template <int W>
__device__ __forceinline__ void insert_pair(const OrbgDeviceCode &code, const BlockSmem<W> &sm,
                                            uint32_t *filter, uint32_t fbits, uint32_t *set,
                                            uint32_t bits, uint32_t lo, uint32_t id)
{
    const uint32_t p = __ldg(code.pairs + id);
    const uint32_t v = sm.h0[p & 0xFFu] ^ sm.h0[p >> 8];
    filter_add(filter, fbits, v);
    const uint32_t x = pair_hash(v), e = slot_tag(x, bits) | (id - lo);
    uint32_t slot = x >> (32u - bits);
    for (;;) {
        const uint32_t old = atomicCAS(set + slot, kEmpty, e);
        if (old == kEmpty)
            return;
        if ((old ^ e) <= kIdMask) {
            /* the same tag: the same syndrome? */
            const uint32_t o = __ldg(code.pairs + lo + (old & kIdMask));
            if (sz(sx(sx(sm.h[p & 0xFFu], sm.h[p >> 8]), sx(sm.h[o & 0xFFu], sm.h[o >> 8])))) {
                atomicMin(set + slot, e);
                return;
            }
        }
        slot = (slot + 1u) & ((1u << bits) - 1u);
    }
}

/* A hit: its query index, its prefix (or kSingle) and its pair (or the
 * 0-based position). */
constexpr uint32_t kSingle = 0xFFFFFFFEu;
struct PairHit {
    uint32_t t, pre, pair;
};

/* s0 (+) the columns of prefix i, whole width. */
template <int W>
__device__ __forceinline__ typename Syn<W>::T prefix_target(const OrbgDeviceCode &code,
                                                            const typename Syn<W>::T *h,
                                                            typename Syn<W>::T s0, uint32_t i)
{
    typename Syn<W>::T v = s0;
    const uint2 r = __ldg(reinterpret_cast<const uint2 *>(code.pre) + i);
    for (uint32_t m = r.x & 0xFFFFu; m; m &= m - 1u)
        v = sx(v, h[(int)__ldg(code.light + (__ffs(m) - 1)) - 1]);
    v = sx(v, sx(h[(int)((r.x >> 16) & 0xFFu) - 1], h[(int)(r.x >> 24) - 1]));
    for (uint32_t y = r.y; y; y >>= 8)
        v = sx(v, h[(int)(y & 0xFFu) - 1]);
    if (code.pext) {
        const uint2 e = __ldg(reinterpret_cast<const uint2 *>(code.pext) + i);
        for (uint32_t y = e.x; y; y >>= 8)
            v = sx(v, h[(int)(y & 0xFFu) - 1]);
        for (uint32_t y = e.y; y; y >>= 8)
            v = sx(v, h[(int)(y & 0xFFu) - 1]);
    }
    return v;
}

/* Query index of prefix i with pair id = p; ORBG_NONE if the pair does not
 * lie after the prefix or the table ends before it. */
__device__ __forceinline__ uint32_t pattern_index(const OrbgDeviceCode &code, uint32_t i,
                                                  uint32_t id, uint32_t p)
{
    const uint2 *pm = reinterpret_cast<const uint2 *>(code.pmeta);
    const uint2 m = __ldg(pm + i);
    const uint32_t q = m.y & 0xFFFFu;
    if ((p & 0xFFu) + 1u <= q)
        return ORBG_NONE;
    const uint32_t end = __ldg(pm + i + 1).x, info = __ldg(code.pinfo + id);
    const uint32_t at = m.x + ((info & 0xFFFFu) - (m.y >> 16));
    if (at >= end)
        return ORBG_NONE;
    /* the first pair of its group after the prefix */
    uint32_t a = info >> 16, b = id;
    while (a < b) {
        const uint32_t mid = (a + b) >> 1;
        if ((uint32_t)(__ldg(code.pairs + mid) & 0xFFu) + 1u > q)
            b = mid;
        else
            a = mid + 1u;
    }
    return __ldg(code.start + at) + (id - a);
}

/* The warp's best of its lanes' hits, in every lane. */
__device__ __forceinline__ PairHit warp_best(const PairHit &mine)
{
    PairHit h;
    h.t = __reduce_min_sync(FULL_MASK, mine.t);
    const int src = __ffs(__ballot_sync(FULL_MASK, mine.t == h.t)) - 1;
    h.pre = __shfl_sync(FULL_MASK, mine.pre, src);
    h.pair = __shfl_sync(FULL_MASK, mine.pair, src);
    return h;
}

/* The best of `best` and the hits of a warp's step: lanes f look for their
 * key v among the first `np` pairs (their keys in `keys`), and the first of a
 * key gives the index with the lane's prefix i.  One lane after the other,
 * each with the whole warp; from kManyHits on (codes of few parity bits) and
 * where the key is the syndrome, every lane for itself and all together: in
 * turn, each would wait for its loads again (60,000 blocks of a (256,248)
 * code, whose look-ups hit in three of five lanes: 173 -> 82 us; of a
 * (256,244) code 173 -> 154, from seven hits on 171; with fewer than four
 * BCH(127,113), a hit a step, gains nothing).  Kept out of line: most steps
 * have none. */
constexpr int kManyHits = 4;
template <int W>
__device__ __noinline__ PairHit resolve_step(const OrbgDeviceCode &code,
                                             const typename Syn<W>::T *h,
                                             typename Syn<W>::T s0, uint32_t i,
                                             const uint32_t *keys, uint32_t v, uint32_t np,
                                             uint32_t f, int lane, PairHit best)
{
    if (W == 1 && __popc(f) >= kManyHits) {
        const uint4 *k4 = reinterpret_cast<const uint4 *>(keys);
        uint32_t id = ORBG_NONE;
#pragma unroll 4
        for (uint32_t k = (np + 3u) / 4u; k-- > 0u;) {
            const uint4 q = k4[k];
            id = q.w == v ? 4u * k + 3u : id;
            id = q.z == v ? 4u * k + 2u : id;
            id = q.y == v ? 4u * k + 1u : id;
            id = q.x == v ? 4u * k : id;
        }
        PairHit mine{ORBG_NONE, i, id};
        if ((f >> lane & 1u) && id < np)
            mine.t = pattern_index(code, i, id, __ldg(code.pairs + id));
        __syncwarp();
        mine = warp_best(mine);
        return mine.t < best.t ? mine : best;
    }
    for (; f; f &= f - 1u) {
        const int src = __ffs(f) - 1;
        const uint32_t key = __shfl_sync(FULL_MASK, v, src);
        const uint32_t pre = __shfl_sync(FULL_MASK, i, src);
        bool found = false;
        for (uint32_t base = 0; base < np && !found; base += 32u) {
            const uint32_t k = base + (uint32_t)lane;
            uint32_t same = __ballot_sync(FULL_MASK, k < np && keys[k] == key);
            for (; same && !found; same &= same - 1u) {
                const uint32_t id = base + (uint32_t)__ffs(same) - 1u;
                const uint32_t p = __ldg(code.pairs + id);
                if (W > 1 && !sz(sx(sx(h[p & 0xFFu], h[p >> 8]),
                                    prefix_target<W>(code, h, s0, pre))))
                    continue;
                found = true;
                const uint32_t t = pattern_index(code, pre, id, p);
                if (t < best.t)
                    best = PairHit{t, pre, id};
            }
        }
    }
    return best;
}

/* The same from a CTA's hash set of the pairs from lo, each lane for itself. */
template <int W>
__device__ __noinline__ uint32_t resolve_hashed(const OrbgDeviceCode &code,
                                                const typename Syn<W>::T *h,
                                                typename Syn<W>::T s0, uint32_t i,
                                                const uint32_t *set, uint32_t bits, uint32_t v,
                                                uint32_t lo, uint32_t *pair)
{
    const uint32_t x = pair_hash(v), tag = slot_tag(x, bits);
    uint32_t slot = x >> (32u - bits);
    typename Syn<W>::T full = s0;
    bool have = W == 1;
    for (;; slot = (slot + 1u) & ((1u << bits) - 1u)) {
        const uint32_t e = set[slot];
        if (e == kEmpty)
            return ORBG_NONE;
        if ((e ^ tag) > kIdMask)
            continue;
        const uint32_t id = lo + (e & kIdMask), p = __ldg(code.pairs + id);
        if (!have) {
            full = prefix_target<W>(code, h, s0, i);
            have = true;
        }
        if (W == 1 ? (syn_key(h[p & 0xFFu]) ^ syn_key(h[p >> 8])) == v
                   : sz(sx(sx(h[p & 0xFFu], h[p >> 8]), full))) {
            *pair = id;
            return pattern_index(code, i, id, p);
        }
    }
}

/* Single positions before `end`: the first whose column is s0.  Thread t of
 * `step` takes positions t, t + step, ...; returns the thread's first hit. */
template <int W>
__device__ __forceinline__ PairHit single_hits(const OrbgDeviceCode &code,
                                               const typename Syn<W>::T *h,
                                               typename Syn<W>::T s0, uint32_t t, uint32_t step,
                                               uint32_t end)
{
    PairHit best{ORBG_NONE, kSingle, 0u};
    for (uint32_t j = t; j < end; j += step)
        if (sz(sx(h[j], s0))) {
            const uint32_t x = __ldg(code.single + j);
            if (x != 0u && x < best.t) {
                best.t = x;
                best.pair = j;
            }
        }
    return best;
}

/*
 * One warp searches band k of its block: the band's pairs from np on go into
 * its filter, then every prefix of the band is looked up, unless `best` or
 * the cap ends the search first.  Returns the best hit, `best` or one found
 * here.  Every pattern before the band's end is covered, so a hit below it
 * is final.  Single positions before the band's are in `best`; only the
 * band's leading sorted positions need be known.
 */
template <int W>
__device__ __forceinline__ PairHit search_band(const OrbgDeviceCode &code,
                                               const BlockSmem<W> &sm,
                                               const typename Syn<W>::T s0, uint32_t cap, int k,
                                               uint32_t np, uint32_t *filter, int lane,
                                               PairHit best)
{
    uint32_t *keys = filter + kWarpFilterBytes / 4u;
    const uint32_t end = code.band_end[k], hi = code.band_pairs[k], npre = code.band_pre[k];
#pragma unroll 1
    for (uint32_t id = np + (uint32_t)lane; id < hi; id += 32u) {
        const uint32_t p = __ldg(code.pairs + id);
        const uint32_t v = sm.h0[p & 0xFFu] ^ sm.h0[p >> 8];
        keys[id] = v;
        filter_add(filter, kWarpFilterBits, v);
    }
    __syncwarp();
    const uint32_t s0w = syn_key(s0);
    const uint2 *gm = reinterpret_cast<const uint2 *>(code.gmeta);
    const uint2 *pre = reinterpret_cast<const uint2 *>(code.pre1);
    if (npre == 0u)
        return best;
    const uint32_t ng = (npre + ORBG_GROUP - 1u) / ORBG_GROUP;
    uint2 nm = __ldg(gm), nr = __ldg(pre + lane);
#pragma unroll 1
    for (uint32_t g = 0; g < ng; g++) {
        const uint2 m = nm, r = nr;
        if (m.x >= end || m.x >= best.t || m.x > cap)
            break;
        /* the next group, loaded while this one is looked up */
        if (g + 1u < ng) {
            nm = __ldg(gm + g + 1u);
            nr = __ldg(pre + (g + 1u) * ORBG_GROUP + (uint32_t)lane);
        }
        const uint32_t i = g * ORBG_GROUP + (uint32_t)lane;
        uint32_t v = s0w;
        const int kmax = (int)(m.y >> 8);
#pragma unroll
        for (int j = 0; j < 8; j++) {
            if (j >= kmax)
                break;
            v ^= sm.h0[(int)(((j < 4 ? r.x : r.y) >> (8 * (j & 3))) & 0xFFu) - 1];
        }
        const uint32_t f =
            __ballot_sync(FULL_MASK, i < npre && filter_has(filter, kWarpFilterBits, v));
        if (f)
            best = resolve_step<W>(code, sm.h, s0, i, keys, v, hi, f, lane, best);
    }
    return best;
}

/* ----------------------------------------------------- step 5: output */

/* Calls flip(received index) for every position of a hit (one thread). */
template <typename F>
__device__ __forceinline__ void pair_flips(const OrbgDeviceCode &code, const PairHit &hit,
                                           const uint8_t *pi, F flip)
{
    if (hit.pre == kSingle) {
        flip(pi[hit.pair]);
        return;
    }
    const uint32_t p = __ldg(code.pairs + hit.pair);
    flip(pi[p & 0xFFu]);
    flip(pi[p >> 8]);
    const uint2 r = __ldg(reinterpret_cast<const uint2 *>(code.pre) + hit.pre);
    for (uint32_t m = r.x & 0xFFFFu; m; m &= m - 1u)
        flip(pi[__ldg(code.light + (__ffs(m) - 1)) - 1]);
    for (uint32_t y = r.x >> 16; y; y >>= 8)
        flip(pi[(y & 0xFFu) - 1u]);
    for (uint32_t y = r.y; y; y >>= 8)
        flip(pi[(y & 0xFFu) - 1u]);
    if (code.pext) {
        const uint2 e = __ldg(reinterpret_cast<const uint2 *>(code.pext) + hit.pre);
        for (uint32_t y = e.x; y; y >>= 8)
            flip(pi[(y & 0xFFu) - 1u]);
        for (uint32_t y = e.y; y; y >>= 8)
            flip(pi[(y & 0xFFu) - 1u]);
    }
}

/* A hit's flips on the hard decision of llr, already in cw: from the LLRs
 * (no read of cw), or, where they are not at hand, on cw itself. */
static __device__ __noinline__ void write_pair_flips(const OrbgDeviceCode &code,
                                                     const PairHit &hit, const uint8_t *pi,
                                                     const float *llr, uint8_t *cw)
{
    pair_flips(code, hit, pi, [=](uint32_t i) { cw[i] = llr[i] > 0.0f ? 0 : 1; });
}
static __device__ __noinline__ void toggle_pair_flips(const OrbgDeviceCode &code,
                                                      const PairHit &hit, const uint8_t *pi,
                                                      uint8_t *cw)
{
    pair_flips(code, hit, pi, [=](uint32_t i) { cw[i] ^= 1; });
}

/* ---------------------------------------------------- the flat table */

/* Flat-table pattern t (1-based): up to ORBG_FLAT_POS positions. */
__device__ __forceinline__ int flat_pos(const uint2 &e, int i)
{
    return (int)(((i < 4 ? e.x : e.y) >> (8 * (i & 3))) & 0xFFu); /* 1-based, 0 = none */
}

/* Flat-table entry t (1-based) or, past the table or the cap, an entry with
 * no positions whose rank count is 0. */
__device__ __forceinline__ uint2 flat_entry(const OrbgDeviceCode &code, uint32_t t, uint32_t cap)
{
    if (t > code.nflat || t > cap)
        return make_uint2(0u, 0u);
    return __ldg(reinterpret_cast<const uint2 *>(code.flat) + (t - 1));
}

/* The step byte of entry e: ranks needed (bits 0-4), largest weight
 * (bits 5-7). */
__device__ __forceinline__ uint32_t flat_step(const uint2 &e) { return e.y >> 24; }

/* Is flat pattern e a hit?  wmax (warp-uniform) bounds its weight.  (An
 * entry with no positions is tested as the zero pattern: callers pass only
 * entries of real queries past query 1.) */
template <int W>
__device__ __forceinline__ bool flat_test(const typename Syn<W>::T *__restrict__ h,
                                          const uint32_t *__restrict__ h0,
                                          const typename Syn<W>::T s0, const uint2 &e, int n,
                                          int wmax = ORBG_FLAT_POS)
{
    typedef typename Syn<W>::T T;
    uint32_t P0 = syn_key(s0);
#pragma unroll
    for (int i = 0; i < ORBG_FLAT_POS; i++) {
        if (i >= wmax)
            break;
        const int q = flat_pos(e, i);
        P0 ^= h0[q - 1];
    }
    if (P0 != 0u)
        return false;
    if (W > 1) {
        T P = s0;
        for (int i = 0; i < ORBG_FLAT_POS; i++) {
            const int q = flat_pos(e, i);
            if (q)
                P = sx(P, h[q - 1]);
        }
        if (!sz(P))
            return false;
    }
    return true;
}

/* Flips of flat pattern t on the hard decision of llr, already in cw. */
template <bool LS>
__device__ __forceinline__ void write_flat_flips(const OrbgDeviceCode &code, uint32_t t,
                                                 const uint8_t *pi, const float *llr, uint8_t *cw)
{
    const uint2 e = __ldg(reinterpret_cast<const uint2 *>(code.flat) + (t - 1));
    for (int i = 0; i < ORBG_FLAT_POS; i++) {
        const int q = flat_pos(e, i);
        if (q == 0)
            break; /* positions come first, zeros after */
        const int idx = pi[q - 1];
        cw[idx] = llr_at<LS>(llr, idx) > 0.0f ? 0 : 1;
    }
}

/* The flat table past its first part, queries from .. code.long_end - 1 in
 * order, by one warp: the first hit, or ORBG_NONE (as flat_test, an entry with
 * no positions is none).  128 queries a step, their entries loaded while the
 * step before is tested: step by step of 32 as the first part, whose ranks are
 * found on the way, a query cost three times as much. */
template <int W>
__device__ __noinline__ uint32_t search_long_flat(const OrbgDeviceCode &code,
                                                  const typename Syn<W>::T *h, const uint32_t *h0,
                                                  typename Syn<W>::T s0, uint32_t from, int lane)
{
    const uint2 *flat = reinterpret_cast<const uint2 *>(code.flat) - 1; /* 1-based */
    const uint32_t end = code.long_end, s0w = syn_key(s0);
    uint2 e[4], next[4];
#pragma unroll
    for (int u = 0; u < 4; u++) {
        const uint32_t t = from + 32u * u + (uint32_t)lane;
        next[u] = t < end ? __ldg(flat + t) : make_uint2(0u, 0u);
    }
#pragma unroll 1
    for (uint32_t base = from; base < end; base += 128u) {
        uint32_t mine = ORBG_NONE;
#pragma unroll
        for (int u = 0; u < 4; u++) {
            e[u] = next[u];
            const uint32_t t = base + 128u + 32u * u + (uint32_t)lane;
            next[u] = t < end ? __ldg(flat + t) : make_uint2(0u, 0u);
        }
#pragma unroll
        for (int u = 3; u >= 0; u--) {
            uint32_t v = s0w;
#pragma unroll
            for (int i = 0; i < ORBG_FLAT_POS; i++)
                v ^= h0[flat_pos(e[u], i) - 1];
            if (v == 0u && (W == 1 || flat_test<W>(h, h0, s0, e[u], 0)))
                mine = base + 32u * u + (uint32_t)lane;
        }
        const uint32_t first = __reduce_min_sync(FULL_MASK, mine);
        if (first != ORBG_NONE)
            return first;
    }
    return ORBG_NONE;
}

/* ------------------------------------------------ one warp, one block */

/*
 * Decode one block with one warp: the flat table, then the bands
 * (search_bands) while no hit is known and the next one starts within
 * `budget`.  A block still open after them is left: its index is
 * appended to heavy[] for decode_block_cta, with its reliability order and
 * starting syndrome in the handover record of the same slot when one is free
 * (hand_cap; bit 63 of the heavy[] entry says so); with heavy NULL hand is
 * its record and the caller takes it up.  Its codeword bytes hold the hard
 * decision by then.  list: key_list_bytes<K>() bytes.  Returns whether the
 * block was finished.  LS: llr
 * points into shared memory (the batched kernel stages it there).
 */
template <int K, int W, bool LS = false>
__device__ bool decode_block_warp(const OrbgDeviceCode &code, const float *__restrict__ llr,
                                  uint8_t *__restrict__ cw_out, uint32_t *__restrict__ q_out,
                                  uint8_t *__restrict__ ab_out, uint32_t cap, uint32_t budget,
                                  unsigned char *__restrict__ bsm, int lane, uint32_t *filter,
                                  uint32_t *list,
                                  unsigned long long *heavy, unsigned long long *heavy_count,
                                  unsigned long long block_index,
                                  unsigned char *hand = nullptr, uint32_t hand_cap = 0)
{
    typedef typename Syn<W>::T T;
    const int n = code.n;
    BlockSmem<W> sm(bsm, n);
    uint32_t key[K]; /* the bits of |L| until they are needed as sort keys */
    bool nan;
    const T s0 = load_block<K, W, LS>(code, llr, key, cw_out, lane, &nan);
    PairHit hit{ORBG_NONE, ORBG_NONE, 0u}; /* prefix NONE: a flat-table hit */
    bool flat_mine = false;
    bool done = true;
    int have = 0; /* leading ranks known; n: all, sorted in full */
    if (!nan && sz(s0)) {
        hit.t = 1u; /* query 1, the zero pattern, is a codeword */
    } else if (!nan) {
        /* the flat table: 32 consecutive queries per step, in query order,
         * so the first step with a hit holds the answer.  Ranks are
         * extracted as the steps need them (one more than needed, so that a
         * tie across the boundary is seen); a tie sorts everything exactly. */
#pragma unroll
        for (int k = 0; k < K; k++)
            key[k] = make_key<K>(key[k], k * 32 + lane);
        sort_lane<K>(key);
        LaneKeys<K> keys(key, list, lane);
        if (lane == 0) {
            sm.h[-1] = szero<T>();
            if (W > 1)
                sm.h0[-1] = 0u;
        }
        uint32_t prev = 0xFFFFFFFFu;
        uint32_t base = 0, tested = 1u, np = 0;
        int k = -1; /* the band; -1: the flat table */
#pragma unroll 1
        for (;;) {
            /* what comes next, and the ranks it needs (one more than needed,
             * so that a tie across the boundary is seen) */
            uint2 e = make_uint2(0u, 0u);
            uint32_t step = 0;
            int upto;
            if (k < 0 && base < code.nflat && base < cap) {
                e = flat_entry(code, base + (uint32_t)lane + 1u, cap);
                /* every entry of a step carries the step byte; entries past
                 * the table are zero */
                step = __reduce_max_sync(FULL_MASK, flat_step(e));
                upto = (int)(step & 31u) + 1;
            } else {
                if (k < 0) {
                    if (cap <= code.nflat)
                        break;
                    tested = code.nflat + 1u;
                }
                for (k++; k < ORBG_BANDS && code.band_end[k] <= tested;)
                    k++;
                if (hit.t < tested || tested > cap)
                    break;
                if (k < ORBG_BANDS && tested <= budget) {
                    upto = (int)code.band_ranks[k] + 1;
                } else {
                    done = false;
                    k = ORBG_BANDS;
                    upto = (int)code.ranks + 1; /* the handover record */
                }
            }
            upto = min(upto, n);
            if (upto > have) {
                /* a tie among the ranks, or more than kMostRanks, sorts
                 * everything exactly */
                if (upto > kMostRanks || extract_ranks<K>(keys, have, upto, &prev, sm.pi)) {
                    make_keys<K, LS>(llr, n, lane, key);
                    sort_block<K, LS>(key, llr, n, lane);
                    build_perm<K, W>(code, key, sm, lane);
                    have = n;
                } else {
                    __syncwarp();
                    perm_ranks<W>(code, have, upto, sm, lane);
                    have = upto;
                }
                __syncwarp();
            }
            if (k < 0) {
                /* 32 consecutive queries in query order: the first step with
                 * a hit holds the answer */
                const uint32_t mine =
                    (e.x | e.y << 8) != 0u &&
                            flat_test<W>(sm.h, sm.h0, s0, e, n, (int)(step >> 5))
                        ? base + (uint32_t)lane + 1u
                        : ORBG_NONE;
                const uint32_t gbest = __reduce_min_sync(FULL_MASK, mine);
                if (gbest != ORBG_NONE) {
                    hit.t = gbest;
                    flat_mine = mine == gbest;
                    break;
                }
                base += 32u;
            } else if (W == 1 && k == 0 && code.long_end != 0u) { /* few rows: one word */
                const uint32_t t = search_long_flat<W>(code, sm.h, sm.h0, s0, tested, lane);
                if (t != ORBG_NONE) {
                    hit.t = t;
                    flat_mine = lane == 0;
                    break;
                }
                tested = code.long_end;
            } else if (k < ORBG_BANDS) {
                if (np == 0u) {
                    uint4 *clear = reinterpret_cast<uint4 *>(filter);
                    for (uint32_t i = (uint32_t)lane; i < kWarpFilterBytes / 16u; i += 32u)
                        clear[i] = make_uint4(0u, 0u, 0u, 0u);
                    __syncwarp();
                }
                hit = warp_best(single_hits<W>(code, sm.h, s0, (uint32_t)lane, 32u,
                                               code.band_ranks[k]));
                hit = search_band<W>(code, sm, s0, cap, k, np, filter, lane, hit);
                np = code.band_pairs[k];
                tested = code.band_end[k];
            } else {
                break;
            }
        }
    }
    if (!done) {
        if (heavy != nullptr) {
            unsigned long long slot = 0;
            if (lane == 0)
                slot = atomicAdd(heavy_count, 1ull);
            slot = __shfl_sync(FULL_MASK, slot, 0);
            const bool keep = slot < (unsigned long long)hand_cap;
            if (keep) {
                unsigned char *rec = hand + slot * ORBG_HANDOVER_BYTES;
                for (int e = lane; e < (int)code.ranks; e += 32)
                    rec[e] = sm.pi[e];
                if (lane == 0)
                    *reinterpret_cast<T *>(rec + 256) = s0;
            }
            if (lane == 0)
                heavy[slot] = block_index | (keep ? 1ull << 63 : 0ull);
        } else {
            for (int e = lane; e < (int)code.ranks; e += 32)
                hand[e] = sm.pi[e];
            if (lane == 0)
                *reinterpret_cast<T *>(hand + 256) = s0;
        }
        __syncwarp();
        return false;
    }
    const bool found = !nan && hit.t <= cap;
    if (found && hit.t > 1u) {
        __syncwarp(); /* after the other lanes' stores of the hard decision */
        if (flat_mine)
            write_flat_flips<LS>(code, hit.t, sm.pi, llr, cw_out);
        else if (hit.pre != ORBG_NONE && lane == 0)
            write_pair_flips(code, hit, sm.pi, llr, cw_out);
    }
    if (lane == 0) {
        *q_out = nan ? 0u : found ? hit.t : cap;
        *ab_out = nan ? 2 : found ? 0 : 1;
    }
    __syncwarp();
    return true;
}

/* The block loaded and sorted by one warp (rare: a block past phase 1's
 * handover records): order, permuted columns and *s0.  Returns 0, 1 for a code
 * word, 2 for a NaN block. */
template <int K, int W>
__device__ __noinline__ int load_and_sort_k(const OrbgDeviceCode &code, const float *llr,
                                            unsigned char *bsm, int lane,
                                            typename Syn<W>::T *s0)
{
    const int n = code.n;
    const BlockSmem<W> sm(bsm, n);
    uint32_t key[K];
    bool nan;
    *s0 = load_block<K, W>(code, llr, key, nullptr, lane, &nan);
    if (nan)
        return 2;
    if (sz(*s0))
        return 1;
    make_keys<K, false>(llr, n, lane, key);
    sort_block<K>(key, llr, n, lane);
    build_perm<K, W>(code, key, sm, lane);
    return 0;
}
template <int W>
__device__ __forceinline__ int load_and_sort(const OrbgDeviceCode &code, const float *llr,
                                             unsigned char *bsm, int lane, typename Syn<W>::T *s0)
{
    return code.n <= 32    ? load_and_sort_k<1, W>(code, llr, bsm, lane, s0)
           : code.n <= 64  ? load_and_sort_k<2, W>(code, llr, bsm, lane, s0)
           : code.n <= 128 ? load_and_sort_k<4, W>(code, llr, bsm, lane, s0)
                           : load_and_sort_k<8, W>(code, llr, bsm, lane, s0);
}

/* ------------------------------------ few prefixes, many pairs: a scan */

/*
 * The CTA's search of an order with code.scan set (the models that come close
 * to ordering by Hamming weight): thousands of pairs, and too few prefixes to
 * pay for inserting them.  The pairs are gone through in their order instead:
 *   - alone, which covers every pattern before the first prefix of a position
 *     (cut_end[0]): the first kScanLead of them, then, where any pair of
 *     columns makes up s0 at all, the others.  Whether one does takes each
 *     thread one comparison a row of pairs, its columns in registers, where a
 *     pair of the list takes ten instructions;
 *   - then with the prefixes' targets (s0 and the prefix's columns) in the
 *     filter and the set, one look-up a pair.  All prefixes of a target stay
 *     in the set: which of them comes first depends on the pair.
 * The empty prefix's index of a pair bounds from below every hit of that pair
 * and later ones.  100,000 blocks of a (255,231) code at 4.5-7 dB and cap
 * 1e5, 32,385 pairs and 45 prefixes: in hash sets of 2,047 pairs 4,400 us,
 * patterns one by one 1,160, pair by pair here 1,650, with the rows 770.
 */
constexpr uint32_t kScanLead = 2048;
template <int W>
__device__ __noinline__ PairHit scan_pairs(const OrbgDeviceCode &code, const BlockSmem<W> sm,
                                           const typename Syn<W>::T s0, uint32_t cap,
                                           uint32_t *filter, uint32_t fbits, uint32_t *set,
                                           uint32_t bits, volatile uint32_t *s_best, int warp,
                                           int lane, int nwarps, PairHit mine)
{
    const uint32_t s0w = syn_key(s0);
    const uint32_t *two = reinterpret_cast<const uint32_t *>(code.pairs);
    auto take = [&](uint32_t pre, uint32_t id, uint32_t p) {
        const uint32_t t = pattern_index(code, pre, id, p);
        if (t < mine.t) {
            mine = PairHit{t, pre, id};
            atomicMin(const_cast<uint32_t *>(s_best), t);
        }
    };
    auto first_of = [&](uint32_t id) {
        return __ldg(code.start + (__ldg(code.pinfo + id) & 0xFFFFu));
    };
    /* 64 pairs a warp step, two a lane; a pair is always the same thread's */
    const uint32_t step = (uint32_t)nwarps * 64u;
    auto alone = [&](uint32_t lo, uint32_t hi) {
#pragma unroll 1
        for (uint32_t base = lo + (uint32_t)warp * 64u; base < hi; base += step) {
            const uint32_t id = base + 2u * (uint32_t)lane;
            const uint32_t p2 = id < hi ? __ldg(two + (id >> 1)) : 0u;
#pragma unroll
            for (uint32_t u = 0; u < 2; u++) {
                const uint32_t p = u ? p2 >> 16 : p2 & 0xFFFFu;
                if ((sm.h0[p & 0xFFu] ^ sm.h0[p >> 8]) == s0w && id + u < hi &&
                    (W == 1 || sz(sx(sx(sm.h[p & 0xFFu], sm.h[p >> 8]), s0))))
                    take(0u, id + u, p);
            }
        }
        __syncthreads();
    };
    const uint32_t lead = min(code.cut_pairs[0], kScanLead / step * step);
    alone(0u, lead);
    if (lead < code.cut_pairs[0] && *s_best >= first_of(lead)) {
        uint32_t col[8];
        bool any = false;
#pragma unroll
        for (int k = 0; k < 8; k++) {
            const uint32_t i = (uint32_t)(k * 32 + lane);
            col[k] = sm.h0[i < code.ranks ? i : 0u];
        }
        for (uint32_t i = (uint32_t)warp; i < code.ranks; i += (uint32_t)nwarps) {
            const uint32_t t = s0w ^ sm.h0[i];
#pragma unroll
            for (int k = 0; k < 8; k++)
                any |= col[k] == t;
        }
        if (__syncthreads_or(any))
            alone(lead, code.cut_pairs[0]);
    }
    if (*s_best < code.cut_end[0] || code.cut_end[0] > cap)
        return mine; /* every pattern before that index is covered (uniform) */
    for (uint32_t i = threadIdx.x; i < (1u << fbits) / 32u; i += blockDim.x)
        filter[i] = 0u;
    for (uint32_t i = threadIdx.x; i < (1u << bits); i += blockDim.x)
        set[i] = kEmpty;
    __syncthreads();
    for (uint32_t i = threadIdx.x; i < code.npre; i += blockDim.x) {
        const uint32_t v = syn_key(prefix_target<W>(code, sm.h, s0, i));
        filter_add(filter, fbits, v);
        const uint32_t x = pair_hash(v);
        uint32_t slot = x >> (32u - bits);
        while (atomicCAS(set + slot, kEmpty, slot_tag(x, bits) | i) != kEmpty)
            slot = (slot + 1u) & ((1u << bits) - 1u);
    }
    __syncthreads();
    const uint32_t end = code.cut_pairs[1];
#pragma unroll 1
    for (uint32_t base = (uint32_t)warp * 64u; base < end; base += step) {
        const uint32_t from = first_of(base);
        if (from >= *s_best || from > cap)
            break;
        const uint32_t id = base + 2u * (uint32_t)lane;
        const uint32_t p2 = id < end ? __ldg(two + (id >> 1)) : 0u;
#pragma unroll 1
        for (uint32_t u = 0; u < 2; u++) {
            const uint32_t p = u ? p2 >> 16 : p2 & 0xFFFFu;
            const uint32_t v = sm.h0[p & 0xFFu] ^ sm.h0[p >> 8];
            if (id + u >= end || !filter_has(filter, fbits, v))
                continue;
            const uint32_t x = pair_hash(v), tag = slot_tag(x, bits);
            for (uint32_t slot = x >> (32u - bits); set[slot] != kEmpty;
                 slot = (slot + 1u) & ((1u << bits) - 1u)) {
                const uint32_t e = set[slot], pre = e & kIdMask;
                if ((e ^ tag) <= kIdMask && sz(sx(sx(sm.h[p & 0xFFu], sm.h[p >> 8]),
                                                  prefix_target<W>(code, sm.h, s0, pre))))
                    take(pre, id + u, p);
            }
        }
    }
    return mine;
}

/* ------------------------------------------------ one CTA, one block */

/*
 * All warps of the CTA decode one block whose hard decision is in cw_out
 * already (its warp wrote it).  Its order comes from the
 * handover record, or warp 0 loads and sorts; all threads then build the
 * subset tables of the light positions and the filter of the block's pairs
 * (several in turn for an order of more than kPairChunk pairs: its cuts, then
 * chunks; scan_pairs takes one of many pairs and few prefixes); then
 * warp w looks up the prefixes of groups w, w + nw, w + 2 nw, ...  Each warp
 * stops at its first group whose floor is at least the shared best (or above
 * the cap): floors never decrease with the group index and the best never
 * increases, so no group that could hold the final best is skipped.
 * pair_sm: pair_smem_bytes(code.chunk) bytes.  SCAN: the code may have scan
 * set (with the call in it, a set of codes that have not lost 1 %).
 */
template <int W, bool SCAN>
__device__ void decode_block_cta(const OrbgDeviceCode &code, const float *__restrict__ llr,
                                 uint8_t *__restrict__ cw_out, uint32_t *__restrict__ q_out,
                                 uint8_t *__restrict__ ab_out, uint32_t cap,
                                 unsigned char *__restrict__ bsm, unsigned char *pair_sm,
                                 uint32_t *s_best, typename Syn<W>::T *s_s0,
                                 int warp, int lane, int nwarps,
                                 const unsigned char *__restrict__ rec = nullptr)
{
    typedef typename Syn<W>::T T;
    const int n = code.n;
    BlockSmem<W> sm(bsm, n);
    uint32_t *mask = reinterpret_cast<uint32_t *>(pair_sm);
    const uint32_t fbits = pair_filter_bits(code.chunk), bits = pair_slot_bits(code.chunk);
    uint32_t *filter = reinterpret_cast<uint32_t *>(pair_sm + kMaskBytes);
    uint32_t *set = filter + (1u << fbits) / 32u;
    if (rec != nullptr) {
        /* phase 1's handover record: the leading part of the block's order
         * that its patterns use, and the starting syndrome; every thread
         * takes a share of the positions */
        for (int i = (int)threadIdx.x; i < (int)code.ranks; i += (int)blockDim.x) {
            const int idx = (int)rec[i];
            sm.pi[i] = (uint8_t)idx;
            const T col = load_col<W>(code.hcol, idx);
            sm.h[i] = col;
            if (W > 1)
                sm.h0[i] = syn_key(col);
        }
        if (threadIdx.x == 0) {
            sm.h[-1] = szero<T>();
            if (W > 1)
                sm.h0[-1] = 0u;
            *s_best = ORBG_NONE;
            *s_s0 = *reinterpret_cast<const T *>(rec + 256);
        }
    } else if (warp == 0) {
        /* not expected to end here (the warp pass finishes such blocks), but
         * exact: a NaN block, or a code word */
        T s0;
        const int what = load_and_sort<W>(code, llr, bsm, lane, &s0);
        if (lane == 0) {
            *s_best = what == 0 ? ORBG_NONE : what == 1 ? 1u : ORBG_NONE - 1u;
            *s_s0 = s0;
        }
    }
    __syncthreads();
    const uint32_t start = *s_best;
    __syncthreads();
    PairHit mine{ORBG_NONE, ORBG_NONE, 0u};
    if (start == ORBG_NONE) {
        const T s0 = *s_s0;
        const uint32_t s0w = syn_key(s0);
        mine = single_hits<W>(code, sm.h, s0, threadIdx.x, blockDim.x, code.ranks);
        if (mine.t != ORBG_NONE)
            atomicMin(s_best, mine.t);
        if (SCAN && code.scan) {
            mine = scan_pairs<W>(code, sm, s0, cap, filter, fbits, set, bits, s_best, warp, lane,
                                 nwarps, mine);
        } else {
            const uint4 light = __ldg(reinterpret_cast<const uint4 *>(code.light));
            for (uint32_t e = threadIdx.x; e < 512u; e += blockDim.x) {
                const uint32_t w0 = e < 256u ? light.x : light.z, w1 = e < 256u ? light.y : light.w;
                uint32_t v = 0;
    #pragma unroll
                for (int b = 0; b < 8; b++) {
                    const int p = (int)(((b < 4 ? w0 : w1) >> (8 * (b & 3))) & 0xFFu);
                    const uint32_t c = sm.h0[p - 1];
                    v ^= e >> b & 1u ? c : 0u;
                }
                mask[e] = v;
            }
            const uint4 *gm = reinterpret_cast<const uint4 *>(code.gmeta);
            const uint2 *pre = reinterpret_cast<const uint2 *>(code.pre);
            /* all pairs at once; or up to one cut after the other, then the rest
             * chunk by chunk */
            uint32_t lo = 0, hi = 0;
            int cut = code.chunk < code.npairs ? 0 : ORBG_CUTS;
    #pragma unroll 1
            for (;;) {
                const uint32_t from = hi;
                uint32_t end = ORBG_NONE, limit = ORBG_NONE;
                bool fresh = cut == 0;
                if (cut < ORBG_CUTS) {
                    hi = code.cut_pairs[cut];
                    end = code.cut_end[cut];
                    /* the last cut's pairs are looked up in full: the chunk ends
                     * with them */
                    limit = ++cut < ORBG_CUTS ? end : ORBG_NONE;
                } else {
                    lo = hi;
                    hi = min(code.npairs, lo + code.chunk);
                    fresh = true;
                }
                if (fresh) {
                    uint4 *clear = reinterpret_cast<uint4 *>(filter);
                    for (uint32_t i = threadIdx.x; i < (1u << fbits) / 128u; i += blockDim.x)
                        clear[i] = make_uint4(0u, 0u, 0u, 0u);
                    clear = reinterpret_cast<uint4 *>(set);
                    for (uint32_t i = threadIdx.x; i < (1u << bits) / 4u; i += blockDim.x)
                        clear[i] = make_uint4(kEmpty, kEmpty, kEmpty, kEmpty);
                }
                __syncthreads();
                for (uint32_t id = from + threadIdx.x; id < hi; id += blockDim.x)
                    insert_pair<W>(code, sm, filter, fbits, set, bits, lo, id);
                __syncthreads();
                /* two groups a warp step: their loads overlap, and the step's
                 * overhead is shared (60 -> 48 warp instructions a group) */
                const uint32_t ng2 = (code.ngroups + 1u) / 2u;
                uint32_t g = (uint32_t)warp;
                uint4 nm = make_uint4(ORBG_NONE, 0u, ORBG_NONE, 0u);
                uint2 nr0 = make_uint2(0u, 0u), nr1 = nr0;
                if (g < ng2) {
                    nm = __ldg(gm + g);
                    nr0 = __ldg(pre + g * 64u + (uint32_t)lane);
                    nr1 = __ldg(pre + g * 64u + 32u + (uint32_t)lane);
                }
    #pragma unroll 1
                for (; g < ng2; g += (uint32_t)nwarps) {
                    const uint4 m = nm;
                    const uint2 r0 = nr0, r1 = nr1;
                    const uint32_t best = *((volatile uint32_t *)s_best);
                    if (m.x >= min(best, limit) || m.x > cap)
                        break;
                    /* the warp's next groups, loaded while these are searched */
                    const uint32_t gn = g + (uint32_t)nwarps;
                    if (gn < ng2) {
                        nm = __ldg(gm + gn);
                        nr0 = __ldg(pre + gn * 64u + (uint32_t)lane);
                        nr1 = __ldg(pre + gn * 64u + 32u + (uint32_t)lane);
                    }
                    const uint32_t i = g * 64u + (uint32_t)lane;
                    uint32_t v0 = s0w ^ mask[r0.x & 0xFFu] ^ mask[256u + ((r0.x >> 8) & 0xFFu)];
                    uint32_t v1 = s0w ^ mask[r1.x & 0xFFu] ^ mask[256u + ((r1.x >> 8) & 0xFFu)];
                    const int kmax = (int)max(m.y & 0xFFu, m.w & 0xFFu);
    #pragma unroll
                    for (int j = 0; j < ORBG_PRE_POS; j++) {
                        if (j >= kmax)
                            break;
                        const uint32_t p0 = j < 2 ? r0.x >> (16 + 8 * j) : r0.y >> (8 * (j - 2));
                        const uint32_t p1 = j < 2 ? r1.x >> (16 + 8 * j) : r1.y >> (8 * (j - 2));
                        v0 ^= sm.h0[(int)(p0 & 0xFFu) - 1];
                        v1 ^= sm.h0[(int)(p1 & 0xFFu) - 1];
                    }
                    if (kmax > ORBG_PRE_POS) {
                        const uint2 *ext = reinterpret_cast<const uint2 *>(code.pext);
                        const uint2 x0 = __ldg(ext + i), x1 = __ldg(ext + i + 32u);
                        for (int j = 0; j < 8; j++) {
                            v0 ^= sm.h0[(int)(((j < 4 ? x0.x : x0.y) >> (8 * (j & 3))) & 0xFFu) - 1];
                            v1 ^= sm.h0[(int)(((j < 4 ? x1.x : x1.y) >> (8 * (j & 3))) & 0xFFu) - 1];
                        }
                    }
                    const bool maybe0 = filter_has(filter, fbits, v0);
                    const bool maybe1 = filter_has(filter, fbits, v1);
                    if (__any_sync(FULL_MASK, maybe0 | maybe1)) {
    #pragma unroll 1
                        for (int w = 0; w < 2; w++) {
                            const uint32_t iw = i + 32u * (uint32_t)w;
                            if (!(w ? maybe1 : maybe0) || iw >= code.npre)
                                continue;
                            uint32_t pair = 0;
                            const uint32_t t = resolve_hashed<W>(code, sm.h, s0, iw, set, bits,
                                                                 w ? v1 : v0, lo, &pair);
                            if (t < mine.t) {
                                mine.t = t;
                                mine.pre = iw;
                                mine.pair = pair;
                                atomicMin(s_best, t);
                            }
                        }
                        __syncwarp();
                    }
                }
                __syncthreads(); /* the filter is free before the next pairs */
                if (hi >= code.npairs ||
                    (end != ORBG_NONE && (*((volatile uint32_t *)s_best) < end || end > cap)))
                    break; /* every pattern before `end` is covered (uniform) */
            }
        }
    }
    __syncthreads();
    const uint32_t best = *s_best;
    const bool is_nan = best == ORBG_NONE - 1;
    const bool hit = !is_nan && best <= cap;
    if (start == ORBG_NONE && hit && mine.t == best)
        toggle_pair_flips(code, mine, sm.pi, cw_out);
    if (warp == 0 && lane == 0) {
        *q_out = is_nan ? 0u : hit ? best : cap;
        *ab_out = is_nan ? 2 : hit ? 0 : 1;
    }
    __syncthreads();
}

/* ----------------------------------------------------------- dispatch */

/* Runtime dispatch on the syndrome width, uniform over the CTA; only widths
 * up to WMAX are instantiated. */
#define ORBG_DISPATCH_W(WMAX, CALL)                                       \
    do {                                                                  \
        const int w_ = code.w32;                                          \
        bool dw_ = false;                                                 \
        if constexpr (WMAX >= 4) {                                        \
            if (w_ > 2) { CALL(4); dw_ = true; }                          \
        }                                                                 \
        if constexpr (WMAX >= 2) {                                        \
            if (!dw_ && w_ == 2) { CALL(2); dw_ = true; }                 \
        }                                                                 \
        if (!dw_) { CALL(1); }                                            \
    } while (0)

}  // namespace orbg_dev
