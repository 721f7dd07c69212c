// DOPH reduction, the first step of the sparse transform (Alg. 3): densified
// one permutation hashing with rotation (Shrivastava and Li).  One hash
// pi(v) = h(Ap, Bp, v) stands for the permutation; its 32-bit range is cut
// into Dp equal bins, bin(v) = (pi(v) * Dp) >> 32 and offset(v) =
// (pi(v) * Dp) mod 2^32; a bin keeps the smallest offset of its items; an
// empty bin takes the value of the first non-empty bin to its right
// (circular) at distance t; an empty set gives t = Dp and value 2^32 - 1.
// The reduced object is the set of Dp tokens (b << 48) | (t << 32) | value.
#include "internal.cuh"

namespace {

constexpr int DP_MAX = 1024, DP_WARPS = 8;

// Warp per set: bin minima by shared-memory atomics, the non-empty bins as a
// bit mask beside them, and each lane finds its bins' nearest non-empty bin at
// or to the right in the mask, a word at a time (with D' = 400 and 59 items the
// next one is 7 bins away on average).  What is left is the write of the
// tokens, 8 D' bytes per set.  500,000 sets, D' = 400: 0.44 ms; 9.9 ms when
// lane 0 walked the 2 D' bins of every set alone.
__global__ void __launch_bounds__(DP_WARPS * 32) k_doph(int64_t n, const int64_t *__restrict__ off,
                                                     const uint32_t *__restrict__ items, int Dp, uint64_t Ap,
                                                     uint64_t Bp, uint64_t *__restrict__ tokens) {
    extern __shared__ uint32_t dsm[];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int nwords = (Dp + 31) >> 5;
    uint32_t *m = dsm + (size_t)wib * (Dp + nwords);  // smallest offset of each bin
    uint32_t *mask = m + Dp;                          // non-empty bins
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = warp; i < n; i += nw) {
        for (int b = lane; b < Dp + nwords; b += 32) m[b] = b < Dp ? 0xFFFFFFFFu : 0u;
        __syncwarp();
        for (int64_t p = off[i] + lane; p < off[i + 1]; p += 32) {
            const uint64_t sc = (uint64_t)mh_hash32(Ap, Bp, items[p]) * (uint64_t)Dp;
            const uint32_t b = (uint32_t)(sc >> 32);
            atomicMin(&m[b], (uint32_t)sc);
            atomicOr(&mask[b >> 5], 1u << (b & 31));
        }
        __syncwarp();
        bool any = false;
        for (int w = lane; w < nwords; w += 32) any = any || mask[w];
        any = __any_sync(0xffffffffu, any);
        for (int b = lane; b < Dp; b += 32) {
            uint64_t t = (uint64_t)Dp, v = 0xFFFFFFFFull;
            if (any) {
                int w = b >> 5;
                uint32_t bits = mask[w] & (0xFFFFFFFFu << (b & 31));
                while (!bits) {  // some word holds a bit
                    w = w + 1 == nwords ? 0 : w + 1;
                    bits = mask[w];
                }
                const int s = 32 * w + __ffs((int)bits) - 1;
                t = (uint64_t)(s >= b ? s - b : s - b + Dp);
                v = m[s];
            }
            tokens[i * Dp + b] = ((uint64_t)b << 48) | (t << 32) | v;
        }
        __syncwarp();  // m and mask are reused by the next set
    }
}

}  // namespace

geek_status doph_reduce(geek_ctx *ctx, int64_t n, const int64_t *off, const uint32_t *items, int Dp, uint64_t Ap,
                        uint64_t Bp, uint64_t *tokens, cudaStream_t st) {
    if (Dp < 1 || Dp > DP_MAX) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "DOPH: 1 <= bins <= 1024");
    if (n == 0) return GEEK_OK;
    const size_t smem = (size_t)DP_WARPS * (Dp + (Dp + 31) / 32) * sizeof(uint32_t);
    GK_CUDA(ctx, cudaFuncSetAttribute(k_doph, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    GK_COUNT();
    k_doph<<<(unsigned)std::min<int64_t>(ceil_div(n, DP_WARPS), (int64_t)ctx->num_sms * 8), DP_WARPS * 32, smem, st>>>(
        n, off, items, Dp, Ap, Bp, tokens);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}
