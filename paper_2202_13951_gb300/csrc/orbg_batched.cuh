/*
 * orbg_batched.cuh -- phase 1 of the batched form.  orbg_batched_inst.cu
 * instantiates it once per (keys per lane, syndrome width) pair; the build
 * compiles those twelve objects in parallel.
 *
 * Phase 1 (orbg_batched_kernel): each warp pulls `grab` blocks at a time
 * from an atomic work queue and decodes each with decode_block_warp, giving
 * it a query budget.  Most blocks finish inside the budget (at high SNR
 * query 1 already decodes).  A block still open when its warp reaches the
 * budget is appended to a heavy list.
 * Phase 2 (orbg_heavy_kernel, orbg_heavy.cuh): each CTA pulls heavy blocks
 * one at a time and decodes each with all its warps (decode_block_cta), so a
 * block that needs up to 1e6 queries is searched by a whole SM instead of a
 * single warp.
 * Both phases compute the exact first hit of the same query order, so the
 * result equals the plain form's block for block.
 *
 * Every launch of phase 1 decodes one decoder variant (keys per lane K,
 * syndrome width W); a mixed-code call sorts its blocks by code and launches
 * per variant, or per code where each code has blocks enough.  ONE: all
 * blocks are one code, passed by value as a kernel parameter (constant bank);
 * otherwise each block's descriptor is read from the device array.
 */
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cuda_pipeline.h>

#include "orbg_decode_block.cuh"
#include "orbg_heavy.cuh"

namespace orbg_batched_impl {

using namespace orbg_dev;

constexpr int kCounters = ORBG_BATCHED_COUNTERS;

/* Resident phase-1 CTAs per SM the register allocation is sized for: four
 * for one code of up to 128 keys and one-word syndromes (64 registers; shared
 * memory allows it), else three.  Measured on 400,000 BCH(127,113) blocks:
 * four 340 us, three 368, two 431; where the descriptor is read per block the
 * kernels spill at 64 (three serving codes, 8,191 blocks: four 190 us, three
 * 170; the four mixed codes with n = 256 at four 2,769 us, at three 2,431, at
 * two 2,541). */
#ifndef ORBG_PHASE1_MIN_CTAS
#define ORBG_PHASE1_MIN_CTAS(K, W, ONE) ((ONE) && (K) < 8 && (W) == 1 ? 4 : 3)
#endif

/* ONE: every block is the code in the kernel's parameters; otherwise each
 * block's code comes from the device array, all of keys per lane K and width
 * W (one decoder variant per launch, the blocks taken from their sort
 * buckets). */
template <int K, int W, bool ONE>
__global__ void __launch_bounds__(256, ORBG_PHASE1_MIN_CTAS(K, W, ONE)) orbg_batched_kernel(
    const OrbgDeviceCode *__restrict__ codes, int ncodes, const int32_t *__restrict__ code_id,
    const int64_t *__restrict__ llr_off, const float *__restrict__ llr, int64_t B, uint32_t cap,
    uint32_t budget, uint8_t *__restrict__ cw, const int64_t *__restrict__ cw_off,
    uint32_t *__restrict__ q, uint8_t *__restrict__ ab, unsigned long long *__restrict__ counters,
    unsigned long long *__restrict__ queue, unsigned long long *__restrict__ heavy,
    const uint32_t *__restrict__ perm,
    unsigned char *__restrict__ hand, uint32_t hand_cap, unsigned long long b_base,
    uint32_t bstride, int grab, int ahead, const uint32_t *__restrict__ range_count,
    int blo, int bhi, const __grid_constant__ OrbgDeviceCode code0)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int nwarps = blockDim.x >> 5;
    unsigned char *bsm = smem + warp * bstride;
    /* two LLR slots per warp: the block being decoded and the next one,
     * copied in asynchronously while the current one is decoded */
    constexpr int kSlot = 32 * K;
    float *ring = reinterpret_cast<float *>(smem + nwarps * bstride) + warp * 2 * kSlot;
    /* the warp's own pairs (search_band) */
    uint32_t *filter = reinterpret_cast<uint32_t *>(smem + nwarps * (bstride + 2 * kSlot * 4) +
                                                  warp * kWarpPairBytes);
    uint32_t *list = reinterpret_cast<uint32_t *>(
        smem + nwarps * (bstride + 2 * kSlot * 4 + kWarpPairBytes) + warp * key_list_bytes<K>());
    /* the dense layout's stride: the set's first code's length */
    const int64_t n0 = ONE && !range_count ? code0.n : codes[0].n;

    /* the queue's slots: all B (< 2^32), or (range_count: the per-bucket
     * counts of the sort into perm) the slots of buckets [blo, bhi) */
    uint32_t slot_lo = 0, slot_hi = (uint32_t)B;
    if (range_count) {
        uint32_t before = 0, inside = 0;
        for (int i = lane; i < bhi; i += 32) {
            const uint32_t c = range_count[i];
            if (i < blo)
                before += c;
            else
                inside += c;
        }
        slot_lo = __reduce_add_sync(FULL_MASK, before);
        slot_hi = slot_lo + __reduce_add_sync(FULL_MASK, inside);
    }
    /* the warp's block sequence: `grab` consecutive queue slots per atomic;
     * with perm (mixed codes) slot i holds the block perm[i], so that the
     * blocks of one decoder variant are decoded together.  The slots' blocks
     * are read once per grab, a lane a slot, and their layout entries
     * prefetched (read block by block, each waited for its slot's load).  A
     * warp that finds the queue empty lets a programmatically dependent
     * launch (the next variant's) start on the SMs this one's last blocks
     * leave idle. */
    constexpr uint32_t kNone = 0xFFFFFFFFu;
    uint32_t pos = 0, end = 0;  /* slots of the grab not yet read */
    int have = 0, next = 0;     /* blocks held in the lanes, and the next one to take */
    uint32_t held = 0;
    auto next_block = [&]() -> uint32_t {
        if (next >= have) {
            if (pos >= end) {
                unsigned long long c = 0;
                if (lane == 0)
                    c = atomicAdd(queue, (unsigned long long)grab);
                c = __shfl_sync(FULL_MASK, c, 0);
                if (c >= (unsigned long long)(slot_hi - slot_lo)) {
                    asm volatile("griddepcontrol.launch_dependents;");
                    return kNone;
                }
                pos = slot_lo + (uint32_t)c;
                end = slot_hi - pos > (uint32_t)grab ? pos + (uint32_t)grab : slot_hi;
            }
            have = (int)min(end - pos, 32u);
            next = 0;
            if (lane < have) {
                held = perm ? __ldg(perm + pos + lane) : pos + (uint32_t)lane;
                if (!ONE && code_id)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(code_id + held));
                if (llr_off)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(llr_off + held));
                if (cw_off)
                    asm volatile("prefetch.global.L1 [%0];" ::"l"(cw_off + held));
            }
            pos += (uint32_t)have;
        }
        return __shfl_sync(FULL_MASK, held, next++);
    };
    /* copies block b's LLRs into the ring's slot; returns its code id */
    auto stage = [&](uint32_t b, int slot) -> int {
        int cid = 0;
        if (b != kNone) {
            cid = !ONE && code_id ? code_id[b] : 0;
            if (cid >= 0 && cid < ncodes) {
                const int n = ONE ? code0.n : codes[cid].n;
                const float *src = llr + (llr_off ? llr_off[b] : (int64_t)b * n0);
#pragma unroll
                for (int k = 0; k < K; k++) {
                    const int i = k * 32 + lane;
                    if (i < n)
                        __pipeline_memcpy_async(ring + slot * kSlot + i, src + i, 4);
                }
            }
        }
        __pipeline_commit();
        return cid;
    };

    /* ahead: the next block is taken and its LLRs copied in while this one is
     * decoded; a batch of few blocks a warp leaves it to the others until
     * this one is done */
    uint32_t b = next_block();
    int slot = 0;
    int cid = stage(b, slot);
    while (b != kNone) {
        uint32_t bn = ahead ? next_block() : kNone;
        int cidn = stage(bn, slot ^ 1);
        __pipeline_wait_prior(1); /* block b's copies have landed */
        __syncwarp();
        uint8_t *out = cw + (cw_off ? cw_off[b] : (int64_t)b * n0);
        const float *l = ring + slot * kSlot;
        if (ONE) {
            decode_block_warp<K, W, true>(code0, l, out, q + b, ab + b, cap, budget, bsm,
                                                    lane, filter, list, heavy, &counters[1],
                                                    b_base + b, hand, hand_cap);
        } else if (cid < 0 || cid >= ncodes) {
            if (lane == 0) {
                q[b] = 0u;
                ab[b] = 2;
            }
        } else {
            /* the block's descriptor is read where it is used (a register
             * copy of it spilled) */
            decode_block_warp<K, W, true>(codes[cid], l, out, q + b, ab + b, cap, budget,
                                                    bsm, lane, filter, list, heavy, &counters[1],
                                                    b_base + b, hand, hand_cap);
        }
        __syncwarp(); /* slot is free before it is refilled */
        if (!ahead) {
            bn = next_block();
            cidn = stage(bn, slot ^ 1);
        }
        b = bn;
        cid = cidn;
        slot ^= 1;
    }
    __pipeline_wait_prior(0);
    /* a launch that may have started before the previous one in its stream
     * ended completes only after it (a no-op for any other launch), so the
     * next ordinary launch sees every phase-1 block finished */
    asm volatile("griddepcontrol.wait;" ::: "memory");
}


/* Shared memory of a phase-1 warp: one block's working set, two LLR slots
 * and its own pairs. */
template <int K> constexpr uint32_t warp_smem_bytes(uint32_t bstride)
{
    return bstride + 2u * 32u * K * (uint32_t)sizeof(float) + kWarpPairBytes +
           key_list_bytes<K>();
}

/* How a phase-1 launch of B blocks is cut: warps per CTA, queue slots per
 * grab, whether warps take blocks ahead, the grid, and how far a warp takes
 * its block.  A batch of few blocks is spread over the SMs and shared out
 * block by block: with the tuned grab of four, 257 blocks of BCH(127,113) ran
 * four after another on 65 warps of nine SMs.  Measured with it and without:
 * three serving codes, 8,191 blocks, 170 -> 121 us.  While phase 2's CTAs are
 * not all busy, a block goes there early: up to two blocks a resident warp
 * after the flat table, up to eight after the first band, past that after
 * both.  us, flat / first band / both: three serving codes, 8,191 blocks (2 a
 * warp) 103 / 105 / 122; BCH(127,113), 257 blocks 34 / 38 / 49; four mixed
 * codes, 33,000 blocks (9) 197 / 175 / 205, 100,000 (27) 460 / 380 / 361;
 * BCH(127,113), 100,000 (21) 189 / 137 / 143, 400,000 (82) 645 / 406 / 345.
 * Both bands pay from 27 and 82 blocks a warp on; where between nine and those
 * is not measured, and just above eight the rule is the slower choice. */
struct Cut {
    int wpc, grab, ahead, grid;
    uint32_t budget;
};
template <typename Kern>
int cut_launch(Kern kern, const OrbgBatchedArgs &a, const OrbgDeviceCode *one,
               uint32_t per_warp, Cut *c)
{
    int dev = 0, sms = 1;
    cudaError_t e;
    if ((e = cudaGetDevice(&dev)) != cudaSuccess ||
        (e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev)) != cudaSuccess)
        return (int)e;
    int wpc = a.warps_per_cta > 0 ? (a.warps_per_cta > 8 ? 8 : a.warps_per_cta) : 8;
    const int64_t spread = (a.B + 2 * sms - 1) / (2 * sms); /* two CTAs an SM */
    if (wpc > spread)
        wpc = (int)spread;
    int rc = orbg_grid_for((const void *)kern, wpc * 32, (size_t)per_warp * wpc, a.ctas_per_sm,
                           &c->grid);
    if (rc != 0)
        return rc;
    const int64_t warps = (int64_t)c->grid * wpc;
    int64_t g = a.grab < 1 ? 1 : a.grab;
    /* eight grabs a warp or more (three serving codes, 50,000 blocks, two 334
     * us, eight 299); one code takes longer grabs, since its blocks search
     * alike: two a warp up to 16 parity bits, whose blocks are short beside a
     * grab's wait (60,000 blocks of a (64,52) code: 90 -> 67), else eight
     * rounded in their favour (50,000 blocks of a (200,180) code at 8-9 dB, one
     * at a time 47, two 31) */
    const int64_t fair = !a.code0            ? a.B / (8 * warps)
                         : a.code0->r <= 16 ? a.B / (2 * warps)
                                            : (a.B + 8 * warps - 1) / (8 * warps);
    if (g > fair)
        g = fair > 0 ? fair : 1;
    c->wpc = wpc;
    c->grab = (int)g;
    c->ahead = a.B > 4 * warps;
    c->budget = a.budget;
    /* a code of few parity bits (long flat table) ends most searches by its
     * first band: it stays, and the others are few enough for phase 2 up to
     * forty blocks a warp.  us, flat / first band / both: a (64,56) code, 5,000
     * blocks 25 / 20 / 19, a (48,38) code, 60,000 43 / 42 / 53, 200,000 82 / 74 /
     * 74, 400,000 140 / 142 / 133, a (256,246) code, 60,000 142 / 93 / 103 */
    const bool few_rows = one != nullptr && one->long_end != 0u;
    if (a.B <= 2 * warps && !few_rows)
        c->budget = a.budget < 1u ? a.budget : 1u;
    else if (a.B <= (few_rows ? 40 : 8) * warps)
        c->budget = a.budget < ORBG_FLAT_MAX + 1u ? a.budget : ORBG_FLAT_MAX + 1u;
    const int64_t need = ((a.B + g - 1) / g + wpc - 1) / wpc;
    if (c->grid > need)
        c->grid = (int)(need > 0 ? need : 1);
    return 0;
}

/* Phase 1 of one decoder variant (K, W): the blocks of sort buckets
 * [blo, bhi) of ss.perm (blo < 0: every block, in order), on its own queue.
 * pdl: the launch may begin while the previous launch in the stream (the
 * previous variant's) finishes its last blocks.  one: all of them are this
 * code. */
template <int K, int W>
int launch_exact_t(const OrbgBatchedArgs &a, const OrbgScratch &ss, unsigned long long *queue,
                   int blo, int bhi, int pdl, const OrbgDeviceCode *one)
{
    const int nk = a.n_max < 32 * K ? a.n_max : 32 * K;
    const uint32_t bstride = block_smem_bytes(nk, W);
    auto k1 = one ? orbg_batched_kernel<K, W, true> : orbg_batched_kernel<K, W, false>;
    Cut c;
    const int rc = cut_launch(k1, a, one, warp_smem_bytes<K>(bstride), &c);
    if (rc != 0)
        return rc;
    const bool sorted = blo >= 0;
    const OrbgDeviceCode c0 = one ? *one : OrbgDeviceCode{};
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)c.grid);
    cfg.blockDim = dim3((unsigned)(c.wpc * 32));
    cfg.dynamicSmemBytes = (size_t)warp_smem_bytes<K>(bstride) * c.wpc;
    cfg.stream = (cudaStream_t)a.stream;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 1 : 0;
    return (int)cudaLaunchKernelEx(
        &cfg, k1, a.d_codes, a.ncodes, a.code_id, a.llr_off, a.llr, a.B, a.cap, c.budget, a.cw,
        a.cw_off, a.q, a.ab, ss.counters, queue, ss.heavy,
        sorted ? (const uint32_t *)ss.perm : (const uint32_t *)nullptr, ss.hand, ss.hand_cap,
        (unsigned long long)a.scratch_base, bstride, c.grab, c.ahead,
        sorted ? (const uint32_t *)ss.count : (const uint32_t *)nullptr, blo, bhi, c0);
}

template <int KMAX, int WMAX, bool ONE>
cudaError_t launch_t(const OrbgBatchedArgs &a)
{
    const uint32_t bstride = block_smem_bytes(a.n_max, a.w32_max);
    const OrbgScratch sc =
        orbg_scratch_layout(a.scratch, a.scratch_B > 0 ? a.scratch_B : a.B, a.ncodes);
    unsigned long long *counters = sc.counters;
    unsigned long long *heavy = sc.heavy;
    cudaStream_t st = (cudaStream_t)a.stream;
    cudaError_t e;
    int rc;
    if (a.stage == 2) {
        /* phase 2 over the open blocks every chunk's phase 1 listed */
        return launch_heavy_t<WMAX, ONE>(a, counters, heavy, sc.hand, false);
    }
    /* this launch's slot: its queue heads, bucket counts and cursors, and
     * its blocks' part of the order array */
    const int slot = a.stage == 1 && a.slot == 1 ? 1 : 0;
    const size_t nc = (size_t)a.ncodes + 1;
    unsigned long long *queue = counters + (slot ? 3 : 0);
    unsigned long long *vqueue = counters + 8 + ORBG_MAX_VARIANTS * slot;
    OrbgScratch ss = sc;
    ss.count = sc.count + 2 * nc * slot;
    ss.cursor = ss.count + nc;
    ss.perm = sc.perm + (a.stage == 1 ? a.scratch_base : 0);
    if (a.stage == 0 || a.first_chunk) {
        if ((e = cudaMemsetAsync(a.scratch, 0, sc.zero_bytes, st)) != cudaSuccess)
            return e;
    } else {
        /* a later chunk: fresh queues and bucket counts in its slot; the
         * open-block list and the phase-2 cursor carry on */
        if ((e = cudaMemsetAsync(queue, 0, sizeof(unsigned long long), st)) != cudaSuccess ||
            (e = cudaMemsetAsync(vqueue, 0, ORBG_MAX_VARIANTS * sizeof(unsigned long long),
                                 st)) != cudaSuccess ||
            (e = cudaMemsetAsync(ss.count, 0, 2 * nc * sizeof(uint32_t), st)) != cudaSuccess)
            return e;
    }
    if constexpr (!ONE) {
        /* per-block codes: one launch per decoder variant, each a kernel of
         * that variant alone, or per code; with several the blocks are first
         * grouped by variant (a counting sort by bucket), and each launch
         * after the first may start while the one before finishes */
        const bool per_code =
            a.var.by_bucket != nullptr && a.ncodes > 1 &&
            a.B >= (int64_t)ORBG_PER_CODE_BLOCKS * a.ncodes;
        const bool sorted = per_code || a.var.n > 1;
        if (sorted && (rc = orbg_launch_code_sort(a.code_id, a.var.d_bucket, a.B, a.ncodes, ss,
                                                  per_code ? a.q : nullptr, a.ab, st)) != 0)
            return (cudaError_t)rc;
        const int launches = per_code ? a.ncodes : a.var.n;
        for (int v = 0; v < launches; v++) {
            if (per_code) {
                const OrbgDeviceCode &one = a.var.by_bucket[v];
                const int k = one.n <= 32 ? 1 : one.n <= 64 ? 2 : one.n <= 128 ? 4 : 8;
                rc = orbg_launch_exact(k, one.w32, a, ss, vqueue + v, v, v + 1, v > 0, &one);
            } else {
                rc = orbg_launch_exact(a.var.k[v], a.var.w[v], a, ss, vqueue + v,
                                       sorted ? a.var.blo[v] : -1, a.var.bhi[v], v > 0, nullptr);
            }
            if (rc != 0)
                return (cudaError_t)rc;
        }
    } else {
        auto k1 = orbg_batched_kernel<KMAX, WMAX, true>;
        Cut c;
        if ((rc = cut_launch(k1, a, a.code0, warp_smem_bytes<KMAX>(bstride), &c)) != 0)
            return (cudaError_t)rc;
        k1<<<c.grid, c.wpc * 32, (size_t)warp_smem_bytes<KMAX>(bstride) * c.wpc, st>>>(
            a.d_codes, a.ncodes, a.code_id, a.llr_off, a.llr, a.B, a.cap, c.budget, a.cw, a.cw_off,
            a.q, a.ab, counters, queue, heavy, nullptr, sc.hand, sc.hand_cap,
            (unsigned long long)a.scratch_base, bstride, c.grab, c.ahead, nullptr, 0, 0,
            *a.code0);
        if ((e = cudaGetLastError()) != cudaSuccess)
            return e;
    }
    /* phase 2 runs whatever the budget: phase 1 also leaves a block open
     * after its last band (with an empty list the launch only reads its
     * length) */
    if (a.stage == 1)
        return cudaSuccess; /* phase 2 comes later, over every chunk's list */
    return launch_heavy_t<WMAX, ONE>(a, counters, heavy, sc.hand, true);
}

/* Phases 1 and 2 for keys-per-lane bound KMAX and syndrome width WMAX: one
 * code (a.code0), or per-block codes. */
template <int KMAX, int WMAX>
int launch_kw(const OrbgBatchedArgs &a)
{
    return a.code0 ? (int)launch_t<KMAX, WMAX, true>(a) : (int)launch_t<KMAX, WMAX, false>(a);
}

}  // namespace orbg_batched_impl
