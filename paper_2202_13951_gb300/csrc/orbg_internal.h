/*
 * orbg_internal.h -- data shared between the host side of the library and
 * its CUDA kernels.
 *
 * The query order (position weights rho_j of the sorted positions; patterns
 * by increasing weight, then Hamming weight w, then positions) is held per
 * code as prefixes and pairs.  A pattern of weight w >= 2 is its prefix P,
 * the first w - 2 positions, and the pair a < b of the last two.  With h_j
 * the parity-check column of sorted position j, it is a hit iff h_a ^ h_b =
 * s0 ^ sum over P of h: the pairs of a block go into a filter or hash set of
 * their syndromes, and one look-up per prefix then tests every pattern the
 * prefix starts, of whatever weight.  A search up to 1,004,225 queries (cap
 * 1e6, n >= 82) makes 15,552 look-ups over 1,640 pairs.  Testing its patterns
 * one by one was bound by the integer pipes: CA-Polar(128,94), 100,000 blocks
 * at 3-6 dB and 119,000 queries a block, took 4,720 us, 12e9 tests; with the
 * look-ups it takes 955 us.
 *
 * Only one pair per syndrome matters, the first in the order (weight, a, b):
 * if the first hit of the order is P + {a, b} and a pair {c, d} before {a, b}
 * has the same syndrome, then exchanging {a, b} for {c, d} (both flipped
 * twice cancel) gives a hit that is lighter, or as heavy with fewer
 * positions, or as heavy and as many and lexicographically smaller.  For the
 * same reason a look-up that finds a pair not wholly after its prefix can
 * be passed over.
 *
 * The prefixes are listed by the least weight m(P) of a pattern they start;
 * the floor of a group of 32, the first query index of that weight, bounds
 * from below every hit of it and later groups, which ends a search.  The
 * index of P + {a, b}: start[] holds, per prefix and group of equally heavy
 * pairs, the index of the first one after P, and the pairs of a group
 * follow in the order of a.
 */
#ifndef ORBG_INTERNAL_H
#define ORBG_INTERNAL_H

#include <stdint.h>

#define ORBG_GROUP 32          /* prefixes per warp step: one per lane */
#define ORBG_MAX_FLIPS 22      /* largest Hamming weight of an order's patterns */
#define ORBG_MAX_LOGISTIC 255  /* deepest logistic weight of a line's order */
#define ORBG_PRE_POS 6         /* positions of a prefix record besides the sixteen lightest */

/* Phase 1 (one warp a block) searches in bands: the pairs of the leading
 * pair groups, and the prefixes that lie before the first group left out.
 * For basic ORBGRAND the bands end after logistic weights 31 and 45 (queries
 * 2,375 and 16,857), with 225 and 484 pairs, 84 and 438 prefixes. */
#define ORBG_BANDS 2
#define ORBG_BAND1_PAIRS 225
#define ORBG_BAND2_PAIRS 500
#define ORBG_PRE1_MAX 1024
/* Phase 2 (a CTA a block) holds up to ORBG_PAIR_CHUNK pairs at a time.  An
 * order of more takes ORBG_SPLIT_CHUNK at a time, and of the first ones the
 * leading ORBG_LEAD_PAIRS alone before the others (the cuts of a search:
 * most blocks end at one of them).  Three-segment model of BCH(127,113),
 * 6,441 pairs, us on 100,000 and 300,000 blocks: all pairs in chunks of 4,095
 * 216 and -, its first 900 before them 180 and 434, both cuts 161 and 360;
 * where one chunk holds all, a cut only repeats look-ups (CA-Polar(128,94)
 * 1,030 -> 1,110 us). */
#define ORBG_PAIR_CHUNK 4095
#define ORBG_SPLIT_CHUNK 2047
#define ORBG_LEAD_PAIRS 900
#define ORBG_CUTS 2
/* An order of many pairs alone (at least phase 1's 500) and few prefixes, up
 * to ORBG_SCAN_PREFIXES and half as many as pairs, is searched the other way
 * round, the prefixes held and the pairs gone through (scan_pairs).  Lines on
 * n = 127, 100,000 blocks, hash sets of pairs / scan, us: J_0 = 9000 (8,001
 * pairs, 51 prefixes) 640 / 332; J_0 = 50 at cap 1e6 (7,952 and 2,384) 303 /
 * 486, since every block that reaches the prefixes inserts them all. */
#define ORBG_SCAN_PREFIXES 2047

/* The flat table: the first `nflat` patterns of the order, 8 bytes each:
 * up to 7 positions, 1-based (0 = unused), then a byte describing the
 * pattern's step of 32: bits 0-4 the number of sorted ranks the step needs
 * (the largest position of that step or an earlier one, at most
 * ORBG_FLAT_RANKS), bits 5-7 the step's largest Hamming weight.  A warp
 * tests 32 consecutive patterns per step before it turns to the bands. */
#define ORBG_FLAT_MAX 256
#define ORBG_FLAT_POS 7
#define ORBG_FLAT_RANKS 31
/* Codes of few parity bits, whose searches are short.  Up to ORBG_FEW_ROWS
 * phase 2 takes at most ORBG_FEW_CHUNK pairs at a time, so that the plain form's
 * CTAs of four warps are not held apart by the pair set's room; up to
 * ORBG_LONG_FLAT_ROWS they go through the first band pattern by pattern (the
 * flat table goes on to its end), since most of a band's look-ups would hit by
 * chance.  Plain form, us, as other codes / so: (40,32), 3,000 and 60,000
 * blocks at 4.5-7 dB, 14.8 and 34 / 9.2 and 27; (64,54), 60,000 blocks 52 / 44,
 * 50,000 at 2-3 dB 172 / 119; with the long table alone 9.5 and 29.7, 48, 132;
 * the chunk and four warps at 60,000 blocks, (64,51) 51 / 42, (128,116) 70 / 61
 * (patterns one by one, 40 to 56, 68 and 104). */
#define ORBG_LONG_FLAT_ROWS 10
#define ORBG_FEW_ROWS 13
#define ORBG_FEW_CHUNK 1023

/* What a kernel needs of one code (passed by value or from a device array). */
struct OrbgDeviceCode {
    const uint32_t *hcol;        /* [n][w32]: column j of H, row i at bit i%32 of word i/32 */
    const uint32_t *hrow;        /* [w32][K][32]: 32 received positions of 32 rows of H, K words
                                  * a row (n <= 32, 64, 128, 256: 1, 2, 4, 8): bit j % 32 of
                                  * entry (i / 32, j / 32, i % 32) is H[i][j] */
    const uint16_t *pairs;       /* [npairs] a0 | b0 << 8, 0-based, by (weight, a, b) */
    const uint32_t *pinfo;       /* [npairs] its group of equally heavy pairs | first pair of the
                                  * group << 16 */
    const uint32_t *pre;         /* [2 * npre, padded to two groups] prefix records, 8 bytes: bit i
                                  * position light[i], then ORBG_PRE_POS further positions,
                                  * 1-based, 0 = none */
    const uint32_t *pext;        /* NULL, or as pre: eight positions past those */
    const uint32_t *pre1;        /* as pre: all positions of a prefix of up to eight */
    const uint32_t *gmeta;       /* [2 * ngroups] floor of the group; the most positions of its
                                  * pre (low byte) and pre1 records (next byte) */
    const uint32_t *pmeta;       /* [2 * (npre + 1)] first entry of the prefix in start[]; its
                                  * last position | the first pair group after it << 16 */
    const uint32_t *start;       /* query index of the first pair of a (prefix, group) */
    const uint32_t *single;      /* [n] query index of each single position, 0 = past the table */
    const uint8_t *light;        /* [16] the lightest positions, 1-based, 0 = none (aligned) */
    uint32_t npairs, npre, ngroups;
    uint32_t band_pairs[ORBG_BANDS]; /* phase 1: pairs of each band, */
    uint32_t band_pre[ORBG_BANDS];   /* prefixes, */
    uint32_t band_ranks[ORBG_BANDS]; /* sorted positions they and the band's patterns take, */
    uint32_t band_end[ORBG_BANDS];   /* and the first query index past the band */
    uint32_t ranks;              /* sorted positions any pattern of the order takes */
    uint32_t chunk;              /* phase 2: pairs (scan: prefixes) held at once; where that is not
                                  * all pairs, */
    uint32_t cut_pairs[ORBG_CUTS]; /* the pairs of each cut, the last one a chunk, */
    uint32_t cut_end[ORBG_CUTS]; /* and the first query index past it */
    uint32_t scan;               /* phase 2 holds the prefixes and goes through the pairs: the
                                  * first cut_pairs[0] alone, which covers the queries before
                                  * cut_end[0], then the first cut_pairs[1] with every prefix */
    const uint32_t *flat;        /* flat-table patterns, 8 bytes each: the first nflat, and up to
                                  * query long_end - 1 if that is not 0 */
    uint32_t nflat, long_end;
    uint32_t max_cap;
    int32_t n;
    int32_t r;
    int32_t w32;                 /* syndrome words: 1, 2 or 4 */
};

/* Host-side table builder (orbg_tables.cpp). */
#ifdef __cplusplus
#include <functional>
#include <vector>
/* The arrays of OrbgDeviceCode, see there. */
struct OrbgTables {
    std::vector<uint16_t> pairs, pgroup; /* pgroup: a pair's group */
    std::vector<uint32_t> pinfo;
    std::vector<uint64_t> pre, pre1, pext;
    std::vector<uint32_t> gmeta, pmeta, start, single;
    uint8_t light[16] = {};
    std::vector<uint8_t> flat;           /* 8 bytes per pattern */
    uint32_t npre = 0, nflat = 0, long_end = 0;
    uint32_t band_pairs[ORBG_BANDS] = {}, band_pre[ORBG_BANDS] = {};
    uint32_t band_ranks[ORBG_BANDS] = {}, band_end[ORBG_BANDS] = {};
    uint32_t ranks = 0, chunk = 0, cut_pairs[ORBG_CUTS] = {}, cut_end[ORBG_CUTS] = {};
    uint32_t scan = 0;
    uint64_t patterns = 0;  /* query indices covered (last index) */
};
/* The tables for the order of increasing reliability weight J0 w + beta W
 * (one-line full ORBGRAND; J0 = 0, beta = 1 is basic ORBGRAND). */
#define ORBG_MAX_LINE 1024
int orbg_build_tables(int n, uint64_t cap, OrbgTables *out, long J0 = 0, long beta = 1);
/* What codes of few parity bits r take instead (ORBG_FEW_ROWS,
 * ORBG_LONG_FLAT_ROWS): smaller chunks of pairs, and the flat table over the
 * first band too, if its patterns fit it. */
void orbg_few_rows(OrbgTables *tb, int n, int r);
/* The m-segment model of Eq. relest_seg: segment i = 1..m covers the
 * sorted positions I[i-1] < j <= I[i] (I[0] = 0, I[m] = n) and position j
 * weighs J[i-1] + beta[i-1] (j - I[i-1]); beta >= 1, J[i-1] >= -beta[i-1]. */
#define ORBG_MAX_SEG 8
#define ORBG_MAX_MODEL (1L << 20) /* largest J or beta of a model */
struct OrbgModel {
    int m;
    int I[ORBG_MAX_SEG + 1];
    long J[ORBG_MAX_SEG];
    long beta[ORBG_MAX_SEG];
};
/* The tables for the m-segment order (reliability weight, then Hamming
 * weight, then positions lexicographically). */
int orbg_build_tables_model(int n, uint64_t cap, const OrbgModel &md, OrbgTables *out);
/* Calls f(t, positions, w) for every pattern of query index t <= count, in
 * no particular order: positions 1-based, ascending. */
void orbg_expand_tables(const OrbgTables &tb, int n, uint64_t count,
                        const std::function<void(uint32_t, const int *, int)> &f);

/* GF(2) helpers on dense 0/1 byte matrices (row-major). */
int orbg_gf2_rank(const uint8_t *M, int rows, int cols);
int orbg_gf2_nullspace(const uint8_t *M, int rows, int cols,
                       std::vector<uint8_t> *basis, int *dim);

/* Kernel launchers (orbg_plain.cu, orbg_batched.cu).  Return a cudaError_t value. */
int orbg_launch_plain(const OrbgDeviceCode &code, const float *llr, int64_t B,
                      uint32_t cap, uint8_t *cw, uint32_t *q, uint8_t *ab,
                      void *stream);
/* One batched call (orbg_batched.cu); buffers on the device.  code0: host
 * copy of code 0's descriptor, or NULL; with code_id == NULL every block is
 * code 0 and the kernels take it from their parameters. */
/* The decoder variants of a code set: keys per lane K (n <= 32, 64, 128,
 * 256: 1, 2, 4, 8) and syndrome words W (1, 2, or 4 for 3-4 words), in the
 * order a mixed-code call's phase 1 takes them.  The device table d_bucket
 * gives each code its sort bucket, numbered so that the codes of one
 * variant hold consecutive buckets [blo, bhi); bucket ncodes collects ids
 * outside the set and belongs to the last variant. */
#define ORBG_MAX_VARIANTS 12
struct OrbgVariants {
    int n;
    int k[ORBG_MAX_VARIANTS], w[ORBG_MAX_VARIANTS];
    int blo[ORBG_MAX_VARIANTS], bhi[ORBG_MAX_VARIANTS];
    const int32_t *d_bucket; /* [ncodes] */
    const OrbgDeviceCode *by_bucket; /* host: the descriptor of each bucket's code, for sets of up
                                      * to ORBG_MAX_VARIANTS codes, else NULL */
};
/* A mixed-code call of at least this many blocks per code of such a set
 * launches phase 1 per code, each with its descriptor in the kernel's
 * parameters, and not per variant with descriptors read from memory block by
 * block.  Measured at 250,000 blocks a code (four codes of three variants,
 * 2,392 -> 2,216 us) and at 25,000 (four of one variant, 685 -> 712: the
 * launches and their ends cost more); the line lies between the two, near
 * their geometric mean. */
#define ORBG_PER_CODE_BLOCKS 65536
struct OrbgBatchedArgs {
    const OrbgDeviceCode *d_codes;
    const OrbgDeviceCode *code0;
    int ncodes, n_max, w32_max;
    OrbgVariants var;            /* the set's decoder variants (mixed-code calls) */
    const int32_t *code_id;
    const int64_t *llr_off;
    const float *llr;
    int64_t B;
    uint32_t cap, budget;
    uint8_t *cw;
    const int64_t *cw_off;
    uint32_t *q;
    uint8_t *ab;
    unsigned long long *scratch;
    int warps_per_cta, ctas_per_sm, grab, heavy_warps;
    uint32_t npairs_max;         /* most pairs phase 2 holds at once for a code of the set */
    uint32_t scan_any;           /* a code of the set has scan */
    void *stream;
    /* Staged calls (the host-buffer pipeline: phase 1 chunk by chunk as the
     * LLRs arrive, then one phase 2 over every chunk's open blocks).
     * stage 0: both phases; 1: phase 1 of one chunk, blocks scratch_base ..
     * scratch_base + B - 1 of the whole batch (the pointers already point at
     * the chunk), first_chunk clears the scratch; 2: phase 2 only, over the
     * whole batch (pointers and B of the whole batch).  scratch_B: the
     * batch's block count the scratch is laid out for (0 = B).  slot (stage
     * 1): the queue and code counts this launch uses (0 or 1); a launch
     * resets its slot's unless it clears the whole scratch. */
    int stage;
    int slot;
    int first_chunk;
    int64_t scratch_base;
    int64_t scratch_B;
};
int orbg_launch_batched(const OrbgBatchedArgs &args);
/* orbg_batched_inst.cu, one per (keys per lane K, syndrome words W): both
 * phases, and phase 1 of that decoder variant alone over sort buckets
 * [blo, bhi) (blo < 0: every block) on `queue` (pdl: the launch may begin
 * while the previous one in the stream finishes; one: all of those blocks are
 * this code, else NULL). */
struct OrbgScratch;
#define ORBG_DECLARE_BATCHED(K, W)                                                   \
    int orbg_launch_batched_k##K##w##W(const OrbgBatchedArgs &a);                    \
    int orbg_launch_exact_k##K##w##W(const OrbgBatchedArgs &a, const OrbgScratch &s, \
                                     unsigned long long *queue, int blo, int bhi, int pdl,  \
                                     const OrbgDeviceCode *one);
ORBG_DECLARE_BATCHED(1, 1) ORBG_DECLARE_BATCHED(1, 2) ORBG_DECLARE_BATCHED(1, 4)
ORBG_DECLARE_BATCHED(2, 1) ORBG_DECLARE_BATCHED(2, 2) ORBG_DECLARE_BATCHED(2, 4)
ORBG_DECLARE_BATCHED(4, 1) ORBG_DECLARE_BATCHED(4, 2) ORBG_DECLARE_BATCHED(4, 4)
ORBG_DECLARE_BATCHED(8, 1) ORBG_DECLARE_BATCHED(8, 2) ORBG_DECLARE_BATCHED(8, 4)
#undef ORBG_DECLARE_BATCHED
/* Device scratch of one batched call over B blocks of a set of ncodes codes,
 * in this order: ORBG_BATCHED_COUNTERS 64-bit counters (0: queue head of
 * slot 0, 1: open-block count, 2: phase-2 cursor, 3: queue head of slot 1,
 * 8 + ORBG_MAX_VARIANTS s + v: the queue head of variant v in slot s); for
 * each of two slots, per-bucket block counts and fill cursors (ncodes + 1
 * uint32 each, the last for code ids outside the set); the list of open
 * blocks (B uint64); the blocks in phase 1's order, grouped by decoder
 * variant (B uint32).  The counters, counts and cursors start at zero.  A
 * phase-1 launch uses one slot's queues and counts, so two launches over
 * different chunks of a batch (the host-buffer pipeline's two decode
 * streams) can run at the same time. */
#define ORBG_BATCHED_COUNTERS (8 + 2 * ORBG_MAX_VARIANTS)
#define ORBG_MAX_CODES 1024      /* codes in one set */
size_t orbg_batched_scratch_bytes(int64_t B, int ncodes);
/* Then, 16-byte aligned, up to ORBG_HANDOVER_MAX handover records: for the
 * i-th block phase 1 leaves open, the leading `ranks` positions of its
 * reliability order (room for 256 bytes: the received index of each sorted
 * position) and its starting syndrome (16 bytes), so that phase 2 need not
 * order the block again.  Blocks past the records are loaded and sorted. */
#define ORBG_HANDOVER_MAX 32768
#define ORBG_HANDOVER_BYTES 272
struct OrbgScratch {
    unsigned long long *counters;
    uint32_t *count, *cursor;     /* slot 0's; slot 1's follow at + 2 (ncodes + 1) */
    unsigned long long *heavy;
    uint32_t *perm;
    unsigned char *hand;          /* handover records */
    uint32_t hand_cap;            /* records available */
    size_t zero_bytes;            /* bytes from the start that must be zero */
};
inline OrbgScratch orbg_scratch_layout(void *base, int64_t B, int ncodes)
{
    OrbgScratch s;
    unsigned char *p = (unsigned char *)base;
    const size_t nc = (size_t)(ncodes > 0 ? ncodes : 0) + 1;
    const size_t b = (size_t)(B > 0 ? B : 0);
    s.counters = (unsigned long long *)p;
    s.count = (uint32_t *)(p + 8 * ORBG_BATCHED_COUNTERS);
    s.cursor = s.count + nc;
    s.zero_bytes = 8 * ORBG_BATCHED_COUNTERS + 16 * nc;
    s.heavy = (unsigned long long *)(p + s.zero_bytes);
    s.perm = (uint32_t *)(s.heavy + b);
    const size_t hoff = ((size_t)((unsigned char *)(s.perm + b) - p) + 15) & ~(size_t)15;
    s.hand = p + hoff;
    s.hand_cap = (uint32_t)(b < ORBG_HANDOVER_MAX ? b : ORBG_HANDOVER_MAX);
    return s;
}
/* Order the blocks of a mixed-code call by the bucket of their code
 * (bucket[code id]; ids outside the set go to bucket ncodes): a counting
 * sort into perm, so that each decoder variant's blocks hold consecutive
 * slots and one launch per variant or code decodes them; with q and ab given,
 * blocks of ids outside the set are written there (0, ORBG_BLOCK_NAN).
 * Returns a cudaError_t. */
int orbg_launch_code_sort(const int32_t *code_id, const int32_t *bucket, int64_t B, int ncodes,
                          const OrbgScratch &s, uint32_t *q, uint8_t *ab, void *stream);
/* orbg_launch_exact_k*w* for keys per lane K and syndrome words W. */
int orbg_launch_exact(int K, int W, const OrbgBatchedArgs &a, const OrbgScratch &s,
                      unsigned long long *queue, int blo, int bhi, int pdl,
                      const OrbgDeviceCode *one);
/* Outputs of the blocks phase 2 decoded, gathered after the last launch of a
 * batch whose other results already went to the host.  At `out` (memory the
 * device writes, here host-mapped) the heavy list's length (uint64).  With
 * to_cw, to_q, to_ab (the caller's output buffers, device-writable host
 * memory laid out as cw, q, ab) every listed block's outputs are written
 * there in place; otherwise `out` also takes, for the list's first `cap`
 * entries, the block index and query count (uint32 pairs), the flag byte,
 * and from orbg_gather_cw_at(cap) the codeword bytes at a stride of n_max.
 * code_id / cw_off NULL: one code of length n0, dense codewords.  Returns a
 * cudaError_t. */
#ifdef __CUDACC__
__host__ __device__
#endif
inline size_t orbg_gather_cw_at(uint32_t cap) { return (16 + 9 * (size_t)cap + 15) & ~(size_t)15; }
inline size_t orbg_gather_bytes(uint32_t cap, int n_max)
{
    return orbg_gather_cw_at(cap) + (size_t)cap * (size_t)n_max;
}
int orbg_launch_heavy_gather(const OrbgDeviceCode *d_codes, const int32_t *code_id, int n0,
                             const int64_t *cw_off, const uint8_t *cw, const uint32_t *q,
                             const uint8_t *ab, const OrbgScratch &s, unsigned char *out,
                             uint32_t cap, int n_max, uint8_t *to_cw, uint32_t *to_q,
                             uint8_t *to_ab, void *stream);
/* The grid of a persistent launch of kern: as many CTAs as are resident, or
 * ctas_per_sm of them on each SM.  Lets launches of kern take the `smem` bytes
 * of dynamic shared memory too: the limit is an attribute of the kernel on its
 * device, which host threads with other sizes share, and is only ever set to
 * the most the device gives, so that no call lowers it between another's
 * setting and launch (which then fails).  Returns a cudaError_t. */
int orbg_grid_for(const void *kern, int threads, size_t smem, int ctas_per_sm, int *grid_out);

/* A named range on the NVTX timeline for the span of a scope (header-only
 * NVTX v3: a no-op unless a profiler such as Nsight Systems is attached). */
#include <nvtx3/nvToolsExt.h>
struct OrbgRange {
    explicit OrbgRange(const char *name) { nvtxRangePushA(name); }
    ~OrbgRange() { nvtxRangePop(); }
    OrbgRange(const OrbgRange &) = delete;
    OrbgRange &operator=(const OrbgRange &) = delete;
};

/* What a launch needs of a code set (orbg_api.cpp owns the struct). */
#include "../../include/orbg.h"
struct OrbgSetView {
    const OrbgDeviceCode *d_codes;
    OrbgDeviceCode code0;        /* host copy of code 0's descriptor */
    int ncodes, n_max, w32_max;
    OrbgVariants var;
    uint32_t npairs_max, scan_any;
    uint32_t cap_min;
    orbg_tuning tuning;
};
int orbg_codeset_view(const orbg_codeset *set, OrbgSetView *out);
int orbg_codeset_lengths(const orbg_codeset *set, std::vector<int> *n_of);
/* Records a cudaError_t for orbg_last_cuda_error; returns the orbg status. */
int orbg_note_cuda_error(int cuda_error);
/* Fitted one-line decoding (orbg_fit.cu): over B one-line model records,
 * present[J_0 + 1] = 1 for every J_0 met, and cid[b] = lut[J_0 + 1]; NaN
 * blocks count as J_0 = 0 and J_0 is held within [-1, top].  present and
 * lut hold top + 2 entries.  Return a cudaError_t. */
int orbg_fit_mark_lines(const int32_t *models, int64_t B, int32_t top, uint8_t *present,
                        void *stream);
/* orbg_fit_models' launch without its argument checks (B >= 1, 1 <= n <=
 * 256, 1 <= lines <= 8, device buffers); returns a cudaError_t. */
int orbg_fit_launch(const float *llr, int64_t B, int n, int lines, int divisible,
                    int32_t *models, void *stream);
int orbg_fit_map_lines(const int32_t *models, int64_t B, int32_t top, const int32_t *lut,
                       int32_t *cid, void *stream);
/* The per-block fitted decoder (orbg_fitted_search_inst.cu, one per keys per
 * lane K): every block fitted (Sec. III-E) and searched in its own order, in
 * four launches; scratch: orbg_fitsearch_scratch_bytes(B) device bytes
 * (counters; the lists of blocks the second, third and fourth launch search;
 * for each open block a handover record of ORBG_FIT_HAND_BYTES: order, model,
 * starting syndrome).
 * Return a cudaError_t value. */
#define ORBG_FIT_HAND_BYTES 384
inline size_t orbg_fitsearch_scratch_bytes(int64_t B)
{
    const size_t b = (size_t)(B > 0 ? B : 0);
    return 64 + 3 * ((4 * b + 15) & ~(size_t)15) + (size_t)ORBG_FIT_HAND_BYTES * b;
}
#define ORBG_DECLARE_FITSEARCH(K)                                                         \
    int orbg_launch_fitsearch_k##K(const OrbgDeviceCode &code, const float *llr, int64_t B, \
                                   uint32_t cap, int lines, int divisible, uint8_t *cw,     \
                                   uint32_t *q, uint8_t *ab, int32_t *models,               \
                                   unsigned char *scratch, void *stream);
ORBG_DECLARE_FITSEARCH(1) ORBG_DECLARE_FITSEARCH(2) ORBG_DECLARE_FITSEARCH(4)
ORBG_DECLARE_FITSEARCH(8)
#undef ORBG_DECLARE_FITSEARCH
int orbg_launch_int_probe(double *lanes_per_clk_per_sm);
int orbg_launch_smem_probe(double *bytes_per_clk_per_sm);
#endif

#endif /* ORBG_INTERNAL_H */
