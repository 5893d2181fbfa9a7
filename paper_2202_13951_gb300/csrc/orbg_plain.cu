/*
 * orbg_plain.cu -- the plain form: one launch, one warp per block in a static
 * grid (Algorithm 1 per block; see orbg_decode_block.cuh).  A block that its
 * warp's bands leave open is searched by the whole CTA once all its warps
 * are through (the CTA's pair set then takes over their shared memory): one
 * warp alone would hold the launch for a search of a million queries.
 */
#include <cuda_runtime.h>
#include <stdint.h>

#include "orbg_decode_block.cuh"

using namespace orbg_dev;

namespace {

/* Warps of a CTA, and the query past which a warp leaves its block to them
 * all (after the first band).  Measured, us a call on 10,000 and 100,000
 * BCH(127,113) blocks: eight warps, first band 45 and 178; both bands 66 and
 * 200; four warps, first band 55 and 186; flat table alone 62 and 221; two
 * warps, both bands 80 and 259.  Four CTAs an SM for one-word syndromes (64
 * registers): 100,000 of those 188 -> 178, 60,000 blocks of a (200,176) code
 * 237 -> 215.  Four warps for codes of few parity bits (ORBG_FEW_ROWS) up to
 * n = 128: their blocks are short, and a CTA stays until its longest one. */
constexpr int kPlainWarps = 8;
constexpr int kPlainFewWarps = 4;
constexpr uint32_t kPlainBudget = ORBG_FLAT_MAX + 1;

template <int K, int W>
__global__ void __launch_bounds__(32 * kPlainWarps, W == 1 ? 4 : 1) orbg_plain_kernel(
    const __grid_constant__ OrbgDeviceCode code, const float *__restrict__ llr, int64_t B,
    uint32_t cap, uint8_t *__restrict__ cw, uint32_t *__restrict__ q, uint8_t *__restrict__ ab,
    uint32_t bstride)
{
    extern __shared__ __align__(16) unsigned char smem[];
    __shared__ uint32_t s_best;
    __shared__ uint4 s_s0;
    __shared__ uint32_t s_open;
    /* an open block's order and syndrome, from its warp to the CTA (loaded and
     * sorted again by one warp while the others wait, 60,000 blocks of a
     * (256,244) code 197 us, 169 with the record) */
    __shared__ __align__(16) unsigned char s_rec[kPlainWarps][ORBG_HANDOVER_BYTES];
    const int warp = threadIdx.x >> 5;
    const int lane = threadIdx.x & 31;
    const int nwarps = blockDim.x >> 5;
    const int64_t b0 = (int64_t)blockIdx.x * nwarps;
    if (threadIdx.x == 0)
        s_open = 0u;
    __syncthreads();
    const int64_t b = b0 + warp;
    if (b < B) {
        const int64_t off = b * (int64_t)code.n;
        unsigned char *own = smem + warp * (bstride + kWarpPairBytes + key_list_bytes<K>());
        const bool done = decode_block_warp<K, W, false>(
            code, llr + off, cw + off, q + b, ab + b, cap, kPlainBudget, own, lane,
            reinterpret_cast<uint32_t *>(own + bstride),
            reinterpret_cast<uint32_t *>(own + bstride + kWarpPairBytes), nullptr, nullptr, 0ull,
            s_rec[warp]);
        if (!done && lane == 0)
            atomicOr(&s_open, 1u << warp);
    }
    __syncthreads();
    for (uint32_t open = s_open; open; open &= open - 1u) {
        const int w = __ffs(open) - 1;
        const int64_t bo = b0 + w;
        const int64_t off = bo * (int64_t)code.n;
        decode_block_cta<W, true>(code, llr + off, cw + off, q + bo, ab + bo, cap, smem, smem + bstride,
                            &s_best, reinterpret_cast<typename Syn<W>::T *>(&s_s0), warp, lane,
                            nwarps, s_rec[w]);
    }
}

template <int K, int W>
cudaError_t launch_plain_t(const OrbgDeviceCode &code, const float *llr, int64_t B, uint32_t cap,
                           uint8_t *cw, uint32_t *q, uint8_t *ab, cudaStream_t st)
{
    const uint32_t bstride = block_smem_bytes(code.n, W);
    const int nw = code.r <= ORBG_FEW_ROWS && K <= 4 ? kPlainFewWarps : kPlainWarps;
    size_t smem = (size_t)(bstride + kWarpPairBytes + key_list_bytes<K>()) * nw;
    const size_t cta = (size_t)bstride + pair_smem_bytes(code.chunk);
    if (smem < cta)
        smem = cta;
    int64_t grid = (B + nw - 1) / nw;
    if (grid > 0x7FFFFFFF)
        return cudaErrorInvalidValue;
    auto k = orbg_plain_kernel<K, W>;
    if (smem > 45 * 1024) { /* with the static part past 48 KB, perhaps */
        int resident;       /* not needed: the grid is the blocks' */
        const int rc = orbg_grid_for((const void *)k, nw * 32, smem, 0, &resident);
        if (rc != 0)
            return (cudaError_t)rc;
    }
    k<<<(unsigned)grid, nw * 32, smem, st>>>(code, llr, B, cap, cw, q, ab, bstride);
    return cudaGetLastError();
}

}  // namespace

int orbg_launch_plain(const OrbgDeviceCode &code, const float *llr, int64_t B, uint32_t cap,
                      uint8_t *cw, uint32_t *q, uint8_t *ab, void *stream)
{
    cudaStream_t st = (cudaStream_t)stream;
    const int n = code.n, w = code.w32;
#define ORBG_PLAIN(KK)                                                            \
    return (int)(w == 1 ? launch_plain_t<KK, 1>(code, llr, B, cap, cw, q, ab, st) \
                 : w == 2 ? launch_plain_t<KK, 2>(code, llr, B, cap, cw, q, ab, st) \
                          : launch_plain_t<KK, 4>(code, llr, B, cap, cw, q, ab, st));
    if (n <= 32) {
        ORBG_PLAIN(1)
    } else if (n <= 64) {
        ORBG_PLAIN(2)
    } else if (n <= 128) {
        ORBG_PLAIN(4)
    } else {
        ORBG_PLAIN(8)
    }
#undef ORBG_PLAIN
}

