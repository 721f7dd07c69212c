// Label = the centre with the most attributes equal to the row's, ties to the
// smallest index: the categorical assignment of Sect. 3.3 (1 - Jaccard of A
// attribute-tagged values falls as the matches rise), for heterogeneous rows
// and for DOPH-reduced sets.
//
// A row meets k centres in A attributes each, but a value of one attribute
// always meets the same centres: every distinct (attribute, value) among the
// centres gets a bit mask of the centres that hold it.  A row then looks its A
// values up in a hash table and adds A masks: lane = 32 centres, the counts
// kept bit-sliced (plane p holds bit p of 32 centres' counts), eight masks at a
// time through a carry-save tree (14 three-input logic operations for 256
// additions), and the largest count and its first centre fall out of the
// planes from the top.  What bounds it is the latency of the two random L2
// reads per attribute (table slot, mask), so the values of a row are looked
// up by 32 lanes at once and the masks are read eight at a time.
// 2,000,000 rows of 18 attributes, k = 196: 0.68 ms (comparing every pair of
// 64-bit values 3.4 ms); 500,000 rows of 400 tokens, k = 425: 4.1 ms (token ids
// by binary search and the posting lists of the Jaccard engine 13.1 ms).
#include "internal.cuh"

namespace {

constexpr int MB_WARPS = 8;
constexpr int MB_IDS = 1024;                  // ids of one warp's rows kept in shared memory
constexpr int64_t MB_MASK_BYTES = 1ll << 30;  // largest mask table (bytes)

struct __align__(16) MbSlot {
    uint64_t value;
    uint32_t attr;  // attribute, 0xFFFFFFFF: empty
    uint32_t id;    // row of the mask table
};

__device__ __forceinline__ uint64_t mb_hash(uint64_t v, uint32_t a) {
    // SplitMix64 finalizer (Steele, Lea and Flood, 2014) of the tagged value
    uint64_t z = v + 0x9e3779b97f4a7c15ull * (uint64_t)(a + 1);
    z = (z ^ (z >> 30)) * 0xbf58476d1ce4e5b9ull;
    z = (z ^ (z >> 27)) * 0x94d049bb133111ebull;
    return z ^ (z >> 31);
}

// owner[s] = 1 + the centre entry e = j A + a that claimed slot s; slot_of[e] =
// the slot of e's (attribute, value).  At most half the slots are ever taken.
__global__ void k_mb_claim(int64_t m, int A, const uint64_t *__restrict__ modes, uint64_t mask,
                           uint32_t *__restrict__ owner, uint32_t *__restrict__ slot_of) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t v = modes[e];
        const uint32_t a = (uint32_t)(e % A);
        for (uint64_t s = mb_hash(v, a) & mask;; s = (s + 1) & mask) {
            uint32_t o = owner[s];
            if (o == 0) o = atomicCAS(&owner[s], 0u, (uint32_t)e + 1u);
            if (o == 0 || ((o - 1) % (uint32_t)A == a && modes[o - 1] == v)) {
                slot_of[e] = (uint32_t)s;
                break;
            }
        }
    }
}

// the finished slots, mask rows numbered in any order
__global__ void k_mb_slots(int64_t nslots, int A, const uint64_t *__restrict__ modes, const uint32_t *__restrict__ owner,
                           unsigned *__restrict__ next, MbSlot *__restrict__ slots) {
    for (int64_t s = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; s < nslots; s += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t o = owner[s];
        MbSlot q{0, 0xFFFFFFFFu, 0};
        if (o) {
            q.value = modes[o - 1];
            q.attr = (o - 1) % (uint32_t)A;
            q.id = atomicAdd(next, 1u);
        }
        slots[s] = q;
    }
}

__global__ void k_mb_masks(int64_t m, int A, int W, const uint32_t *__restrict__ slot_of,
                           const MbSlot *__restrict__ slots, uint32_t *__restrict__ masks) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = e / A;
        atomicOr(&masks[(int64_t)slots[slot_of[e]].id * W + (j >> 5)], 1u << (j & 31));
    }
}

// carry-save adder: a + b + c = l + 2 h, bit by bit
__device__ __forceinline__ void csa(uint32_t &h, uint32_t &l, uint32_t a, uint32_t b, uint32_t c) {
    h = (a & b) | (a & c) | (b & c);
    l = a ^ b ^ c;
}

// A warp takes 32 / LG rows at a time, LG lanes (a power of two, at least the
// W mask words or 32) per row; rows of more than 32 words take several rounds.
// PL planes hold counts up to A < 2^PL.  hist (nullable): rows by match count.
template <int PL>
__global__ void __launch_bounds__(32 * MB_WARPS) k_mb_assign(int64_t n, int A, int64_t k, int W, int LG, int RW,
                                                              const uint64_t *__restrict__ attrs,
                                                              const MbSlot *__restrict__ slots, uint64_t mask,
                                                              const uint32_t *__restrict__ masks,
                                                              int32_t *__restrict__ labels,
                                                              unsigned long long *__restrict__ hist) {
    __shared__ uint32_t s_ids[MB_WARPS][MB_IDS];
    __shared__ unsigned s_hist[MB_IDS + 1];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    uint32_t *ids = s_ids[w];
    if (hist) {
        for (int e = threadIdx.x; e <= A; e += blockDim.x) s_hist[e] = 0;
        __syncthreads();
    }
    const int sub = lane & (LG - 1), rr = lane / LG;  // word lane, row of the warp's RW
    const uint32_t gmask = (LG == 32 ? 0xFFFFFFFFu : ((1u << LG) - 1u)) << (rr * LG);
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t nwarps = (int64_t)gridDim.x * MB_WARPS;
    for (int64_t i0 = ((int64_t)blockIdx.x * MB_WARPS + w) * RW; i0 < n; i0 += nwarps * RW) {
        // the rows' values that some centre holds, as mask rows
        int cnt = 0;  // of this lane's row
        for (int r = 0; r < RW; r++) {
            const int64_t i = i0 + r;
            int c = 0;
            for (int a0 = 0; a0 < A; a0 += 32) {
                const int a = a0 + lane;
                uint32_t id = 0xFFFFFFFFu;
                if (a < A && i < n) {
                    const uint64_t v = attrs[i * A + a];
                    for (uint64_t s = mb_hash(v, (uint32_t)a) & mask;; s = (s + 1) & mask) {
                        const uint4 q = reinterpret_cast<const uint4 *>(slots)[s];
                        if (q.z == 0xFFFFFFFFu) break;
                        if (q.z == (uint32_t)a && q.x == (uint32_t)v && q.y == (uint32_t)(v >> 32)) {
                            id = q.w;
                            break;
                        }
                    }
                }
                const uint32_t b = __ballot_sync(0xffffffffu, id != 0xFFFFFFFFu);
                if (id != 0xFFFFFFFFu) ids[r * A + c + __popc(b & lt)] = id;
                c += __popc(b);
            }
            if (rr == r) cnt = c;
        }
        __syncwarp();
        const int64_t i = i0 + rr;
        const bool row = rr < RW && i < n;
        const uint32_t *my = ids + (rr < RW ? rr * A : 0);
        int most = cnt;  // the longest list of the warp's rows
        if (RW > 1) most = __reduce_max_sync(0xffffffffu, cnt);
        int best = -1, bj = 0;
        for (int w0 = 0; w0 < W; w0 += 32) {
            const int word = w0 + sub;
            const bool live = row && word < W;
            uint32_t ones = 0, twos = 0, fours = 0, P[PL];
#pragma unroll
            for (int p = 0; p < PL; p++) P[p] = 0;
            for (int q0 = 0; q0 < most; q0 += 8) {
                uint32_t m[8];
#pragma unroll
                for (int u = 0; u < 8; u++)
                    m[u] = live && q0 + u < cnt ? masks[(int64_t)my[q0 + u] * W + word] : 0u;
                uint32_t ta, tb, tc, td, fa, fb, e8;
                csa(ta, ones, ones, m[0], m[1]);
                csa(tb, ones, ones, m[2], m[3]);
                csa(fa, twos, twos, ta, tb);
                csa(tc, ones, ones, m[4], m[5]);
                csa(td, ones, ones, m[6], m[7]);
                csa(fb, twos, twos, tc, td);
                csa(e8, fours, fours, fa, fb);
#pragma unroll
                for (int p = 3; p < PL; p++) {
                    const uint32_t t = P[p] & e8;
                    P[p] ^= e8;
                    e8 = t;
                }
            }
            P[0] = ones;
            if (PL > 1) P[1] = twos;
            if (PL > 2) P[2] = fours;
            // the largest count of the words' centres, from the top plane down
            const int64_t left = k - (int64_t)word * 32;
            uint32_t cand = !live ? 0u : (left >= 32 ? 0xFFFFFFFFu : (1u << left) - 1u);
            int cb = 0;
#pragma unroll
            for (int p = PL - 1; p >= 0; p--) {
                const uint32_t t = cand & P[p];
                if (__ballot_sync(0xffffffffu, t != 0) & gmask) {
                    cand = t;
                    cb |= 1 << p;
                }
            }
            const uint32_t have = __ballot_sync(0xffffffffu, cand != 0) & gmask;
            const int src = have ? __ffs((int)have) - 1 : lane;
            const int first = __shfl_sync(0xffffffffu, word * 32 + __ffs((int)cand) - 1, src);
            if (have && cb > best) {
                best = cb;
                bj = first;
            }
        }
        if (row && sub == 0) {
            labels[i] = bj;
            if (hist) atomicAdd(&s_hist[best], 1u);
        }
        __syncwarp();
    }
    if (hist) {
        __syncthreads();
        for (int e = threadIdx.x; e <= A; e += blockDim.x)
            if (s_hist[e]) atomicAdd(&hist[e], (unsigned long long)s_hist[e]);
    }
}

uint64_t mb_slots(int64_t k, int A) {
    uint64_t s = 64;
    while (s < 2ull * (uint64_t)k * (uint64_t)A) s <<= 1;
    return s;
}

}  // namespace

// The mask table grows with k^2 A / 8 bytes; above its limit (1 GB, far more
// than L2, so that each row would read its masks from HBM) the callers keep
// their direct forms.
bool match_bits_eligible(int64_t k, int A) {
    return k > 0 && A > 0 && A <= MB_IDS && (double)k * A * (double)(4 * ceil_div(k, 32)) <= (double)MB_MASK_BYTES;
}

// labels[i] = argmax_j #{a : attrs[i][a] == modes[j][a]}, ties to the smallest j
// (attrs n x A, modes k x A, attribute by attribute); hist (nullable, A + 1
// counters, zeroed by the caller): rows by their largest match count.  *done is
// false, and nothing has run, where there is no room for the tables.
geek_status match_bits_assign(geek_ctx *ctx, Scratch &scr, int64_t n, int A, const uint64_t *attrs, int64_t k,
                              const uint64_t *modes, int32_t *labels, unsigned long long *hist, bool *done,
                              cudaStream_t st) {
    const int64_t m = k * A;
    const int W = (int)ceil_div(k, 32);
    const uint64_t ns = mb_slots(k, A);
    uint32_t *owner, *slot_of, *masks;
    unsigned *next;
    MbSlot *slots;
    *done = true;
    GK_TRY(scr.alloc(&next, 1));
    GK_TRY(scr.try_alloc(&masks, (size_t)m * W, done));
    if (*done) GK_TRY(scr.try_alloc(&owner, ns, done));
    if (*done) GK_TRY(scr.try_alloc(&slots, ns, done));
    if (*done) GK_TRY(scr.try_alloc(&slot_of, m, done));
    if (!*done) return GEEK_OK;
    GK_CUDA(ctx, cudaMemsetAsync(owner, 0, sizeof(uint32_t) * ns, st));
    GK_CUDA(ctx, cudaMemsetAsync(masks, 0, sizeof(uint32_t) * (size_t)m * W, st));
    GK_CUDA(ctx, cudaMemsetAsync(next, 0, sizeof(unsigned), st));
    const int gm = grid_for(m, 256, ctx->num_sms);
    GK_COUNT();
    k_mb_claim<<<gm, 256, 0, st>>>(m, A, modes, ns - 1, owner, slot_of);
    GK_COUNT();
    k_mb_slots<<<grid_for((int64_t)ns, 256, ctx->num_sms), 256, 0, st>>>((int64_t)ns, A, modes, owner, next, slots);
    GK_COUNT();
    k_mb_masks<<<gm, 256, 0, st>>>(m, A, W, slot_of, slots, masks);
    GK_LAUNCH(ctx);
    int LG = 1;
    while (LG < W && LG < 32) LG <<= 1;
    const int RW = std::max(1, std::min(32 / LG, MB_IDS / A));
    const unsigned grid = (unsigned)std::min<int64_t>(ceil_div(n, (int64_t)RW * MB_WARPS), (int64_t)ctx->num_sms * 6);
    GK_COUNT();
    if (A < 32)
        k_mb_assign<5><<<grid, 32 * MB_WARPS, 0, st>>>(n, A, k, W, LG, RW, attrs, slots, ns - 1, masks, labels, hist);
    else if (A < 512)
        k_mb_assign<9><<<grid, 32 * MB_WARPS, 0, st>>>(n, A, k, W, LG, RW, attrs, slots, ns - 1, masks, labels, hist);
    else
        k_mb_assign<11><<<grid, 32 * MB_WARPS, 0, st>>>(n, A, k, W, LG, RW, attrs, slots, ns - 1, masks, labels, hist);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}
