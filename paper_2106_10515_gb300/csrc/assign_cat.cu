// Central vectors and assignment for categorical and set data (Sect. 3.3):
//  - heterogeneous rows: unified categorical attributes (per table, the
//    packed key of the numeric E2LSH part; then the tokens), per-attribute
//    mode as central vector, distance 1 - Jaccard = most matching attributes;
//  - sparse sets: central vector = items present in more than half of the
//    members, distance 1 - |A n C| / |A u C| compared exactly as fractions.
#include <algorithm>

#include "internal.cuh"

namespace {

int G(geek_ctx *ctx, int64_t work) { return grid_for(std::max<int64_t>(work, 1), 256, ctx->num_sms); }

// attrs[i][a]: a < L -> numeric key of table a, else token a - L
__global__ void k_build_attrs(int64_t n, int L, int ncat, const uint64_t *__restrict__ num_key,
                              const uint32_t *__restrict__ tok, uint64_t *__restrict__ attrs) {
    const int A = L + ncat;
    const int64_t total = n * A;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = e / A;
        const int a = (int)(e % A);
        attrs[e] = a < L ? num_key[(int64_t)a * n + i] : (uint64_t)tok[i * ncat + (a - L)];
    }
}

// mode of attribute a over seed j's members: most frequent value, ties to the
// smallest (one thread per (seed, attribute); quadratic in the seed size)
// rep (nullable): the first member, in the seed's ascending order, holding
// the mode value
__global__ void k_modes(int64_t k, int A, const int64_t *__restrict__ soff, const int32_t *__restrict__ sids,
                        const uint64_t *__restrict__ attrs, uint64_t *__restrict__ modes, int32_t *__restrict__ rep) {
    const int64_t total = k * A;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = e / A;
        const int a = (int)(e % A);
        const int64_t s = soff[j], t = soff[j + 1];
        uint64_t best = 0;
        int64_t bc = 0;
        int32_t br = -1;
        for (int64_t p = s; p < t; p++) {
            const uint64_t v = attrs[(int64_t)sids[p] * A + a];
            int64_t c = 0;
            for (int64_t q = s; q < t; q++) c += attrs[(int64_t)sids[q] * A + a] == v;
            if (c > bc || (c == bc && v < best)) {
                bc = c;
                best = v;
                br = sids[p];
            }
        }
        modes[e] = best;
        if (rep) rep[e] = br;
    }
}

// flags[g] = 1 where bucket g (global id, in table l's canonical order) starts
// a new numeric E2LSH tuple: the table keys of heterogeneous rows put the
// numeric tuple first, so equal numeric tuples form runs of buckets.
__global__ void k_num_run_flags(int64_t nb, int64_t base, const int64_t *__restrict__ boff,
                                const uint32_t *__restrict__ members, const uint64_t *__restrict__ num_key_l,
                                int64_t *__restrict__ flags) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nb; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t g = base + r;
        int64_t f = 1;
        if (r > 0) f = num_key_l[members[boff[g]]] != num_key_l[members[boff[g - 1]]];
        flags[g] = f;
    }
}

// modes as a user sees them: per table, the rank of the mode's numeric tuple
// among the table's distinct numeric tuples (via the bucket of the member
// that holds it); then the mode tokens
__global__ void k_mode_out(int64_t k, int A, int L, int64_t n, const uint64_t *__restrict__ modes,
                           const int32_t *__restrict__ rep, const int32_t *__restrict__ obj_bucket,
                           const int64_t *__restrict__ tbase, const int64_t *__restrict__ excl,
                           const int64_t *__restrict__ flags, int64_t *__restrict__ out) {
    const int64_t total = k * A;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (int64_t)gridDim.x * blockDim.x) {
        const int a = (int)(e % A);
        if (a < L) {
            // runs started at or before g, less the one at the table's start
            const int64_t g = tbase[a] + obj_bucket[(int64_t)a * n + rep[e]];
            out[e] = excl[g] + flags[g] - 1 - excl[tbase[a]];
        } else {
            out[e] = (int64_t)modes[e];
        }
    }
}

// label = argmax_j #{a : attrs[i][a] == modes[j][a]}, ties to the smallest j
constexpr int CAT_TILE = 64;
constexpr int CAT_MAXA = 32;
__global__ void __launch_bounds__(256) k_assign_cat(int64_t n, int A, int64_t k, const uint64_t *__restrict__ attrs,
                                                    const uint64_t *__restrict__ modes, int32_t *__restrict__ labels,
                                                    unsigned long long *__restrict__ hist) {
    __shared__ uint64_t ms[CAT_TILE * CAT_MAXA];
    __shared__ unsigned s_hist[CAT_MAXA + 1];
    if (threadIdx.x <= CAT_MAXA) s_hist[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    uint64_t x[CAT_MAXA];
    for (int a = 0; a < CAT_MAXA; a++) x[a] = (i < n && a < A) ? attrs[i * A + a] : 0;
    int bm = -1, bj = -1;
    for (int64_t j0 = 0; j0 < k; j0 += CAT_TILE) {
        __syncthreads();
        const int tn = (int)min((int64_t)CAT_TILE, k - j0);
        for (int e = threadIdx.x; e < tn * A; e += blockDim.x) ms[(e / A) * CAT_MAXA + e % A] = modes[(j0 + e / A) * A + e % A];
        __syncthreads();
        for (int jj = 0; jj < tn; jj++) {
            int m = 0;
#pragma unroll
            for (int a = 0; a < CAT_MAXA; a++)
                if (a < A) m += x[a] == ms[jj * CAT_MAXA + a];
            if (m > bm) {
                bm = m;
                bj = (int)(j0 + jj);
            }
        }
    }
    if (i < n) {
        labels[i] = bj;
        if (hist && bm >= 0) atomicAdd(&s_hist[bm], 1u);
    }
    __syncthreads();
    if (hist && threadIdx.x <= A && s_hist[threadIdx.x])
        atomicAdd(&hist[threadIdx.x], (unsigned long long)s_hist[threadIdx.x]);
}

// ---- set data --------------------------------------------------------------

// member weight of each (group, member) entry = size of the member's set
__global__ void k_group_w(int64_t m, const int32_t *__restrict__ gmem, const int64_t *__restrict__ soff,
                          int64_t *__restrict__ w) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < m; p += (int64_t)gridDim.x * blockDim.x)
        w[p] = soff[gmem[p] + 1] - soff[gmem[p]];
}

__global__ void k_group_of(int64_t ng, const int64_t *__restrict__ goff, int32_t *__restrict__ gid) {
    for (int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; g < ng; g += (int64_t)gridDim.x * blockDim.x)
        for (int64_t p = goff[g]; p < goff[g + 1]; p++) gid[p] = (int32_t)g;
}

__global__ void k_group_expand(int64_t m, const int32_t *__restrict__ gid, const int32_t *__restrict__ gmem,
                               const int64_t *__restrict__ woff, const int64_t *__restrict__ soff,
                               const uint32_t *__restrict__ sids, uint64_t *__restrict__ pairs) {
    for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < m; p += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t g = (uint64_t)gid[p];
        const int32_t s = gmem[p];
        int64_t o = woff[p];
        for (int64_t q = soff[s]; q < soff[s + 1]; q++) pairs[o++] = (g << 32) | sids[q];
    }
}

__global__ void k_group_keep(const int64_t *__restrict__ nruns, const int64_t *__restrict__ prs,
                             const uint64_t *__restrict__ pairs, const int64_t *__restrict__ goff,
                             int64_t *__restrict__ keep, int64_t *__restrict__ cnt) {
    const int64_t nr = *nruns;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nr; r += (int64_t)gridDim.x * blockDim.x) {
        const int64_t len = prs[r + 1] - prs[r];
        const int64_t g = (int64_t)(pairs[prs[r]] >> 32);
        const bool kp = 2 * len > goff[g + 1] - goff[g];
        keep[r] = kp;
        if (kp) atomicAdd((unsigned long long *)&cnt[g], 1ull);
    }
}

__global__ void k_group_emit(const int64_t *__restrict__ nruns, const int64_t *__restrict__ prs,
                             const uint64_t *__restrict__ pairs, const int64_t *__restrict__ keep,
                             const int64_t *__restrict__ pos, uint32_t *__restrict__ out) {
    const int64_t nr = *nruns;
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nr; r += (int64_t)gridDim.x * blockDim.x)
        if (keep[r]) out[pos[r]] = (uint32_t)(pairs[prs[r]] & 0xFFFFFFFFu);
}

// heavy items: up to 64 * JX_HW of the items with the longest posting lists
// are counted by bitmasks instead of posting lists
constexpr int JX_HW = 3;

// item -> centres inverted index helpers
__global__ void k_centre_pairs(int64_t k, const int64_t *__restrict__ coff, const uint32_t *__restrict__ citems,
                               uint64_t *__restrict__ pairs) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < k; j += (int64_t)gridDim.x * blockDim.x)
        for (int64_t p = coff[j]; p < coff[j + 1]; p++) pairs[p] = ((uint64_t)citems[p] << 32) | (uint64_t)j;
}


__global__ void k_item_key(int64_t m, const uint64_t *__restrict__ pairs, uint64_t *__restrict__ ikey) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < m; q += (int64_t)gridDim.x * blockDim.x)
        ikey[q] = pairs[q] >> 32;
}



__global__ void k_light_flags(int64_t nr, const int64_t *__restrict__ rs, const int64_t *__restrict__ is_heavy,
                              int64_t *__restrict__ lrun, int64_t *__restrict__ lent) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nr; r += (int64_t)gridDim.x * blockDim.x) {
        const bool light = !is_heavy[r];
        lrun[r] = light;
        lent[r] = light ? rs[r + 1] - rs[r] : 0;
    }
}

__global__ void k_light_emit(int64_t nr, const int64_t *__restrict__ rs, const uint64_t *__restrict__ ikey,
                             const uint64_t *__restrict__ pairs, const int64_t *__restrict__ is_heavy,
                             const int64_t *__restrict__ lrun_pos, const int64_t *__restrict__ lent_pos,
                             uint32_t *__restrict__ litem, int64_t *__restrict__ loff, uint32_t *__restrict__ lcentre,
                             const int64_t *__restrict__ nlent, int64_t nlight) {
    for (int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; r < nr; r += (int64_t)gridDim.x * blockDim.x) {
        if (is_heavy[r]) continue;
        const int64_t p = lrun_pos[r];
        litem[p] = (uint32_t)ikey[rs[r]];
        loff[p] = lent_pos[r];
        int64_t o = lent_pos[r];
        for (int64_t q = rs[r]; q < rs[r + 1]; q++) lcentre[o++] = (uint32_t)(pairs[q] & 0xFFFFFFFFu);
    }
    if (blockIdx.x == 0 && threadIdx.x == 0) loff[nlight] = *nlent;
}

__global__ void k_iota_rows(int64_t n, int32_t *__restrict__ rows, unsigned long long *__restrict__ cnt) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        rows[i] = (int32_t)i;
    if (blockIdx.x == 0 && threadIdx.x == 0) *cnt = (unsigned long long)n;
}

// item of each listed run (first entry's key)
__global__ void k_run_items(int nh, const int64_t *__restrict__ runs, const int64_t *__restrict__ rs,
                            const uint64_t *__restrict__ ikey, uint32_t *__restrict__ out) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nh; q += gridDim.x * blockDim.x)
        out[q] = (uint32_t)ikey[rs[runs[q]]];
}

// heavy items: bit b of the HW-word mask stands for the item hv_item[i] with
// hv_bit[i] = b (hv_item ascending); -1 when x is not heavy
__device__ __forceinline__ int heavy_bit(uint32_t x, const uint32_t *__restrict__ hv_item,
                                         const int16_t *__restrict__ hv_bit, int nheavy) {
    int lo = 0, hi = nheavy;
    while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (hv_item[mid] < x) lo = mid + 1;
        else hi = mid;
    }
    return (lo < nheavy && hv_item[lo] == x) ? hv_bit[lo] : -1;
}

template <int W>
__global__ void k_heavy_masks(int64_t k, const int64_t *__restrict__ coff, const uint32_t *__restrict__ citems,
                              const uint32_t *__restrict__ hv_item, const int16_t *__restrict__ hv_bit, int nheavy,
                              int HW, uint64_t *__restrict__ cmask, int32_t *__restrict__ clen) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < k; j += (int64_t)gridDim.x * blockDim.x) {
        uint64_t m[W] = {};
        for (int64_t p = coff[j]; p < coff[j + 1]; p++) {
            const int b = heavy_bit(citems[p], hv_item, hv_bit, nheavy);
            if (b >= 0) m[b >> 6] |= 1ull << (b & 63);
        }
        for (int w = 0; w < HW; w++) cmask[j * HW + w] = m[w];
        clen[j] = (int32_t)(coff[j + 1] - coff[j]);
    }
}

// Jaccard assignment: warp per set.  Intersections with heavy items come
// from bitmasks; light items go through the inverted index into a per-warp
// counter array (cleared after use).  Every centre is then scored exactly:
// J_j = inter / (|A| + |C_j| - inter), compared by cross-multiplication.
// (The dense path: every centre is scanned per set.  It serves the sets
// with more items than the tiled kernels take;
// rows lists them, na_fix >= 0 replaces |A| by a fixed size.)
template <int MW>  // mask words per centre
__global__ void __launch_bounds__(256) k_assign_jaccard(
    int64_t n, const int64_t *__restrict__ off, const uint32_t *__restrict__ items, int64_t k,
    const int32_t *__restrict__ clen, const uint64_t *__restrict__ cmask, const uint32_t *__restrict__ hv_item,
    const int16_t *__restrict__ hv_bit, int nheavy, const uint32_t *__restrict__ post_item,
    const int64_t *__restrict__ post_off, int64_t n_post_items, const uint32_t *__restrict__ post_centre,
    int32_t *__restrict__ counts, int32_t *__restrict__ labels, const int32_t *__restrict__ rows,
    const unsigned long long *__restrict__ n_rows, int na_fix) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    int32_t *cnt = counts + warp * k;
    if (rows) n = (int64_t)*n_rows;
    for (int64_t ii = warp; ii < n; ii += nw) {
        const int64_t i = rows ? (int64_t)rows[ii] : ii;
        const int64_t s = off[i], e = off[i + 1];
        const int64_t na = na_fix >= 0 ? na_fix : e - s;
        uint64_t am[MW] = {};
        // light items: binary search in the sorted item list of the index
        for (int64_t p = s + lane; p < e; p += 32) {
            const uint32_t it = items[p];
            const int hb = heavy_bit(it, hv_item, hv_bit, nheavy);
            if (hb >= 0) {
#pragma unroll
                for (int w = 0; w < MW; w++)
                    if (hb >> 6 == w) am[w] |= 1ull << (hb & 63);
                continue;
            }
            int64_t lo = 0, hi = n_post_items;
            while (lo < hi) {
                const int64_t mid = (lo + hi) >> 1;
                if (post_item[mid] < it) lo = mid + 1;
                else hi = mid;
            }
            if (lo < n_post_items && post_item[lo] == it)
                for (int64_t q = post_off[lo]; q < post_off[lo + 1]; q++) atomicAdd(&cnt[post_centre[q]], 1);
        }
#pragma unroll
        for (int w = 0; w < MW; w++)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) am[w] |= __shfl_xor_sync(0xffffffffu, am[w], o);
        __syncwarp();
        __threadfence_block();
        int64_t bn = -1, bd = 1;
        int bj = 0x7FFFFFFF;
        for (int64_t j = lane; j < k; j += 32) {
            int64_t in = cnt[j];
#pragma unroll
            for (int w = 0; w < MW; w++) in += __popcll(am[w] & cmask[j * MW + w]);
            cnt[j] = 0;
            const int64_t un = na + clen[j] - in;
            const int64_t num = un ? in : 0, den = un ? un : 1;
            if (bj == 0x7FFFFFFF || num * bd > bn * den) {
                bn = num;
                bd = den;
                bj = (int)j;
            }
        }
        // warp argmax: larger fraction, then smaller index
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const int64_t on = __shfl_xor_sync(0xffffffffu, bn, o);
            const int64_t od = __shfl_xor_sync(0xffffffffu, bd, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            bool take;
            if (oj == 0x7FFFFFFF) take = false;
            else if (bj == 0x7FFFFFFF) take = true;
            else {
                const int64_t l = on * bd, r = bn * od;
                take = l > r || (l == r && oj < bj);
            }
            if (take) {
                bn = on;
                bd = od;
                bj = oj;
            }
        }
        if (lane == 0) labels[i] = bj == 0x7FFFFFFF ? -1 : bj;
        __syncwarp();
    }
}

// Exact Jaccard argmax, tiled over the centres; a warp per set, warps
// independent of one another.  Per tile of `kt` centres every item of the set
// reads the part of its posting list (centres containing the item, ascending)
// that falls in the tile and adds one to the warp's counter of each centre
// there (packed 8- or 16-bit counters in shared memory: a counter counts the
// set's light items in one centre, at most MAXI), so the counters plus the
// heavy items' bitmask give |A n C_j|.
//
// Visiting every (set, centre) pair is what a plain form pays for: scoring a
// pair costs about 15 operations, a set meets 8,192 centres per tile, and
// the few hundred most frequent items alone give 9 of 10 counter increments.
// So there are two passes:
//  k_jac_prune (every set): the JX_MW * 64 most frequent items stay out of
//    the counters.  A centre beats or ties the best fraction bn / bd so far
//    only if |A n C| >= bn (|A| + |C|) / (bn + bd), so its counter is at least
//    that (with the tile's smallest |C|) less the set's number of frequent
//    items: the warp tests the counters of a 16-byte load against this
//    threshold with one add and mask per word and scores the few that pass
//    exactly (64-bit cross products, larger fraction then smaller index; with
//    no positive J the label is 0).  The centre of a tile's largest counter
//    gives the first bound; a tile met while the threshold is not positive, or
//    so near the mean counter that most centres would be scored, is taken
//    again at the end, and if it still is (a set unlike every centre), the set
//    goes to the second pass.  200,000 sets of 60 of 700 items, k = 12,299: this pass
//    8.7 ms with the sign alone, 3.9 with the mean, the second pass 10.0 either way;
//    2M sets of 59 of 64,000 items: 40.7 and 41.2, 23.
//  k_jac_count (those sets): only the most frequent items stay out, 64 to 64
//    JX_HW of them (jx_heavy_words), and every centre is scored, lane per centre
//    (k_jac_count8: thread per four centres, eight sets).
// Sets with more than MAXI items are listed for the dense path.
// 2,000,000 sets of 59 items against 46,553 centres (mean 58 items): the
// counters get 3,200 increments per set instead of 28,600, and the two passes
// take 41 + 22 ms; scoring every pair took 173 ms.  500,000 DOPH rows of 400
// tokens against 425 centres: 4.5 + 5.0 ms, before 31 ms.

// centres from which the second pass scores by blocks (k_jac_count8): k = 3,020 0.99 ms by
// warps, 1.29 by blocks; 4,279 0.090, 0.129; 5,831 4.11, 3.79; 6,393 5.21, 4.69; 7,762 1.06, 0.79
constexpr int JX_BLOCKS = 5120;
constexpr int JX_WARPS = 8;
constexpr int JX_THREADS = 32 * JX_WARPS;
constexpr int JX_MW = 8;  // mask words of the frequent items k_jac_prune leaves out
// NARROW: sets of at most 128 items, 8-bit counters, tiles of up to 8192
// centres; otherwise up to 512 items, 16-bit counters, tiles of up to 4096
// (8 KB of counters per warp either way; fewer when k is smaller).
template <bool NARROW> struct Jx {
    static constexpr int KT = NARROW ? 8192 : 4096;  // centres per tile, at most
    static constexpr int MAXI = NARROW ? 128 : 512;  // items per set on the tiled path
    static constexpr int LG = NARROW ? 2 : 1;        // log2 counters per word
    static constexpr int CBITS = 32 >> LG;
    static constexpr uint32_t CMASK = NARROW ? 0xFFu : 0xFFFFu;
    static constexpr uint32_t ONES = NARROW ? 0x01010101u : 0x00010001u;
    static constexpr uint32_t TOP = NARROW ? 0x80u : 0x8000u;
    static constexpr int STEP = 128 << LG;           // counters per warp-wide 16-byte load
};

// the largest set: max over i of off[i + 1] - off[i]
__global__ void k_max_len(int64_t n, const int64_t *__restrict__ off, unsigned long long *__restrict__ out) {
    unsigned long long m = 0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, (unsigned long long)(off[i + 1] - off[i]));
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0 && m) atomicMax(out, m);
}

// tile_off[r * (ntiles + 1) + t]: the first entry of posting list r whose
// centre is in tile t or later (ntiles + 1 entries per list)
__global__ void k_tile_offsets(int64_t nr, const int64_t *__restrict__ post_off,
                               const uint32_t *__restrict__ post_centre, int ntiles, int kt,
                               int32_t *__restrict__ tile_off) {
    const int64_t tot = nr * (ntiles + 1);
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < tot; e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = e / (ntiles + 1);
        const int t = (int)(e % (ntiles + 1));
        const uint64_t lim = (uint64_t)t * kt;
        int64_t lo = post_off[r], hi = post_off[r + 1];
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if ((uint64_t)post_centre[mid] < lim) lo = mid + 1;
            else hi = mid;
        }
        tile_off[e] = (int32_t)lo;
    }
}

// tile_min[t] = the smallest |C| among the centres of tile t (block per tile)
__global__ void __launch_bounds__(256) k_tile_min_len(int64_t k, int kt, const int32_t *__restrict__ clen,
                                                      int32_t *__restrict__ tile_min) {
    __shared__ int s_min;
    if (threadIdx.x == 0) s_min = INT32_MAX;
    __syncthreads();
    const int64_t c0 = (int64_t)blockIdx.x * kt, c1 = min(k, c0 + kt);
    int m = INT32_MAX;
    for (int64_t c = c0 + threadIdx.x; c < c1; c += 256) m = min(m, clen[c]);
    atomicMin(&s_min, m);
    __syncthreads();
    if (threadIdx.x == 0) tile_min[blockIdx.x] = s_min;
}

// posting entries as centre indices within their tile
__global__ void k_tile_local(int64_t m, const uint32_t *__restrict__ post_centre, int kt, uint16_t *__restrict__ out) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        out[e] = (uint16_t)(post_centre[e] % (uint32_t)kt);
}

// lut[item] for items up to the largest in any centre: -2 - rank for one of
// the 64 JX_MW most frequent items, else its posting list (>= 0), -1 for an
// item no centre holds
__global__ void k_item_lut(int64_t nlight, const uint32_t *__restrict__ litem, int32_t *__restrict__ lut) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < nlight; e += (int64_t)gridDim.x * blockDim.x)
        lut[litem[e]] = (int32_t)e;
}
__global__ void k_freq_lut(int nfreq, const uint32_t *__restrict__ fq_item, const int16_t *__restrict__ fq_bit,
                           int32_t *__restrict__ lut) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nfreq; q += gridDim.x * blockDim.x)
        lut[fq_item[q]] = -2 - (int32_t)fq_bit[q];
}
// posting list of each frequent item by rank (ranks below nheavy have none)
__global__ void k_freq_list(int nfreq, int nheavy, const int64_t *__restrict__ fq_run, const int16_t *__restrict__ fq_bit,
                            const int64_t *__restrict__ lrun_pos, int32_t *__restrict__ fq_list) {
    for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < nfreq; q += gridDim.x * blockDim.x)
        fq_list[fq_bit[q]] = fq_bit[q] < nheavy ? -1 : (int32_t)lrun_pos[fq_run[q]];
}

// Mask words of the heaviest items (ord: by posting list) that pay in the second
// pass.  64 more items in the mask cost a load and a popcount per centre, and save
// a set the counter increments of those it holds, about k sum (len / k)^2 when sets
// resemble centres.  Second pass with one, two and three words, the sum for the
// second word in brackets: 200,000 sets of 60 of 300 items, k = 674 (2.9) 1.00, 0.91
// and 0.75 ms; of 100 of 600, k = 605 (2.5) 1.24, 1.22, 1.07; of 60 of 500, k = 3,057 (1.06)
// 3.08, 3.45, 3.28.  With more than a tile of centres they pay earlier: 300,000 of 60 of
// 500, k = 12,796 (1.07) 21.2, 20.4, 18.8; 200,000 of 40 of 400, k = 10,420 (0.72) 8.6, 8.2, 7.8;
// of 60 of 700, k = 12,299 (0.58) 9.97, 10.15, 9.86; 2M sets, k = 46,553 (0.28) 22.9, 24.3, 27.4.
// Wide sets, whose loop over the items costs more: 100,000 of 300 of 2,000, k = 177 (2.5)
// 1.14, 1.45, 1.46; of 300 of 1,200, k = 1,864 (4.9) 1.79, 1.94, 1.83.
int jx_heavy_words(const std::vector<int64_t> &rs, const std::vector<int32_t> &ord, int nfreq, int64_t k, bool narrow) {
    if (!narrow) return 1;
    int words = 1;
    for (; words < JX_HW && 64 * words < nfreq; words++) {
        double sum = 0.0;
        for (int q = 64 * words; q < std::min(nfreq, 64 * words + 64); q++) {
            const double len = (double)(rs[ord[q] + 1] - rs[ord[q]]) / (double)k;
            sum += len * len;
        }
        if (sum < (k > Jx<true>::KT ? 0.65 : 1.5)) break;
    }
    return words;
}

// how the kernels find an item: the table when the items are small numbers
// (n_lut entries), else binary searches
struct JxIndex {
    const int32_t *lut;
    int64_t n_lut;
    const uint32_t *fq_item;  // frequent items ascending, their ranks
    const int16_t *fq_bit;
    int nfreq;
    const uint32_t *post_item;  // items with posting lists, ascending
    int64_t n_post_items;
    __device__ __forceinline__ int32_t find(uint32_t it) const {
        if (lut) return (int64_t)it < n_lut ? lut[it] : -1;
        const int hb = heavy_bit(it, fq_item, fq_bit, nfreq);
        if (hb >= 0) return -2 - hb;
        int64_t lo = 0, hi = n_post_items;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (post_item[mid] < it) lo = mid + 1;
            else hi = mid;
        }
        return lo < n_post_items && post_item[lo] == it ? (int32_t)lo : -1;
    }
};

struct JxArgs {
    int64_t n;  // sets
    const int64_t *off;
    const uint32_t *items;
    int na_fix;
    int64_t k;
    int kt, ntiles;
    const int32_t *clen, *tile_min, *tile_off;
    const uint16_t *post_local;
    JxIndex X;
    int32_t *labels;
};

// Counts one tile: every item of the warp's set adds one to the counter of
// each centre of its posting list there.  The lanes take 32 items at a time.
// Ranges of JX_LONG entries and more are walked one after the other, lane per
// entry.  A prefix sum turns the shorter ones into one run of entries, walked 32
// at a time with every lane busy (a range is 16 entries on average), at six
// shuffles a step to find each lane's range.  With those steps for long ranges too
// the passes over 200,000 sets of 40 of 400 items, k = 10,420, took 22.1 ms, 8.9
// this way; over 2M sets of 59 of 64,000, k = 46,553: 81.5 and 63.6.  Lines of 32 and
// 64 measured the same, but for 100 of 600 items, k = 339: 1.5 and 1.8 ms.
// Returns the lane's largest (count << 16 | counter) it produced, and adds the
// entries of the lane's items to sum.
constexpr int JX_LONG = 32;
template <class C>
__device__ __forceinline__ uint32_t jx_count(uint32_t *cw, const int32_t *ridx, int ni, int t, const JxArgs &A,
                                             int &sum) {
    const int lane = threadIdx.x & 31, ld = A.ntiles + 1;
    uint32_t lm = 0;
    for (int q0 = 0; q0 < ni; q0 += 32) {
        const int32_t r = q0 + lane < ni ? ridx[q0 + lane] : -1;
        int ps = 0, len = 0;
        if (r >= 0) {
            ps = A.tile_off[(int64_t)r * ld + t];
            len = A.tile_off[(int64_t)r * ld + t + 1] - ps;
        }
        sum += len;
        auto add = [&](uint32_t cc) {
            const int sh = (cc & ((1 << C::LG) - 1)) * C::CBITS;
            const uint32_t old = atomicAdd(&cw[cc >> C::LG], 1u << sh);
            lm = max(lm, (((old >> sh) & C::CMASK) << 16) + 65536u + cc);
        };
        for (uint32_t m = __ballot_sync(0xffffffffu, len >= JX_LONG); m; m &= m - 1) {
            const int src = __ffs((int)m) - 1;
            const int at = __shfl_sync(0xffffffffu, ps, src), ln = __shfl_sync(0xffffffffu, len, src);
#pragma unroll 4
            for (int e = lane; e < ln; e += 32) add(A.post_local[at + e]);
        }
        if (len >= JX_LONG) len = 0;
        int inc = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, inc, o);
            if (lane >= o) inc += y;
        }
        const int tot = __shfl_sync(0xffffffffu, inc, 31);
        const int ex = inc - len, base = ps - ex;
#pragma unroll 2
        for (int e0 = 0; e0 < tot; e0 += 32) {
            const int e = e0 + lane;
            int src = 0;  // the last range starting at or before entry e
#pragma unroll
            for (int o = 16; o > 0; o >>= 1)
                if (__shfl_sync(0xffffffffu, ex, src + o) <= e) src += o;
            const int at = __shfl_sync(0xffffffffu, base, src) + e;
            if (e < tot) add(A.post_local[at]);
        }
    }
    return lm;
}

// the best centre of a set: larger fraction n / d, then smaller index
struct JxBest {
    uint32_t n = 0, d = 1;
    int j = 0x7FFFFFFF;
    // |A| + |C| < 2^16: both cross products fit 32 bits
    __device__ __forceinline__ void push(uint32_t on, uint32_t od, int oj) {
        const uint32_t l = on * d, r = n * od;
        if (l > r || (l == r && oj < j)) {
            n = on;
            d = od;
            j = oj;
        }
    }
    __device__ __forceinline__ void warp_merge() {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1)
            push(__shfl_xor_sync(0xffffffffu, n, o), __shfl_xor_sync(0xffffffffu, d, o),
                 __shfl_xor_sync(0xffffffffu, j, o));
    }
    // the smallest |A n C| that still beats or ties it, |C| >= cmin
    __device__ __forceinline__ uint32_t need(uint32_t na, uint32_t cmin) const {
        return max((n * (na + cmin) + n + d - 1) / (n + d), 1u);
    }
};

template <bool NARROW>
__global__ void __launch_bounds__(JX_THREADS, 3) k_jac_prune(JxArgs A, const uint64_t *__restrict__ fmask, int FW,
                                                             int32_t *__restrict__ ovf_rows,
                                                             unsigned long long *__restrict__ n_ovf,
                                                             int4 *__restrict__ hard_rows,
                                                             unsigned long long *__restrict__ n_hard) {
    using C = Jx<NARROW>;
    extern __shared__ uint4 jx_smem[];
    __shared__ unsigned long long s_am[JX_WARPS][JX_MW];  // the set's frequent items
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nv = A.kt / C::STEP;  // 16-byte loads per lane and tile
    uint4 *c4 = jx_smem + (size_t)w * nv * 32;
    uint32_t *cw = reinterpret_cast<uint32_t *>(c4);
    int32_t *ridx = reinterpret_cast<int32_t *>(jx_smem + (size_t)JX_WARPS * nv * 32) + w * C::MAXI;
    unsigned long long *am = s_am[w];
    for (int v = lane; v < nv * 32; v += 32) c4[v] = make_uint4(0u, 0u, 0u, 0u);
    const int64_t nwarps = (int64_t)gridDim.x * JX_WARPS;
    for (int64_t i = (int64_t)blockIdx.x * JX_WARPS + w; i < A.n; i += nwarps) {
        const int64_t s0 = A.off[i], e0 = A.off[i + 1];
        if (e0 - s0 > C::MAXI) {
            if (lane == 0) ovf_rows[atomicAdd(n_ovf, 1ull)] = (int32_t)i;
            continue;
        }
        const int ni = (int)(e0 - s0);
        const uint32_t na = (uint32_t)(A.na_fix >= 0 ? A.na_fix : ni);
        __syncwarp();
        if (lane < JX_MW) am[lane] = 0ull;
        __syncwarp();
        // the items: frequent ones into the mask, the others' posting lists
        int mine = 0;
#pragma unroll 2
        for (int p = lane; p < ni; p += 32) {
            const int32_t r = A.X.find(A.items[s0 + p]);
            ridx[p] = r;
            if (r < -1) {
                const int hb = -2 - r;
                atomicOr(&am[hb >> 6], 1ull << (hb & 63));
                mine++;
            }
        }
        const int hcnt = __reduce_add_sync(0xffffffffu, mine);  // frequent items of the set
        __syncwarp();
        JxBest best;  // the same on every lane
        auto score = [&](int64_t c, uint32_t l, JxBest &b) {
            uint32_t in = l;
            for (int h = 0; h < FW; h++) in += __popcll(am[h] & fmask[c * FW + h]);
            if (in) b.push(in, na + (uint32_t)A.clen[c] - in, (int)c);
        };
        // tiles met without a positive threshold, taken again at the end
        uint64_t again = 0;
        bool hard = false;
        // a threshold at most two deviations above the mean counter (as of a Poisson count)
        auto weak = [](int need, float entries, int64_t centres) {
            const float d = (float)need * (float)centres - entries;
            return d <= 0.0f || d * d <= 4.0f * entries * (float)centres;
        };
        float total = 0.0f;
        for (int tt = 0, t = 0; !hard; tt++) {
            const bool second = tt >= A.ntiles;
            if (!second) {
                t = tt;
            } else {
                if (!again) break;
                t = __ffsll((long long)again) - 1;
                again &= again - 1;
            }
            const int64_t c0 = (int64_t)t * A.kt;
            const uint32_t cmin = (uint32_t)A.tile_min[t];
            int need = (int)best.need(na, cmin) - hcnt;
            if (second && weak(need, total, A.k)) {
                hard = true;
                break;
            }
            int sum = 0;
            const uint32_t lm = __reduce_max_sync(0xffffffffu, jx_count<C>(cw, ridx, ni, t, A, sum));
            __syncwarp();
            bool low = false;
            if (!second) {
                sum = __reduce_add_sync(0xffffffffu, sum);
                total += (float)sum;
                low = weak(need, (float)sum, min((int64_t)A.kt, A.k - c0));
            }
            if (low) {
                // the centre of the tile's largest counter as a first bound
                if (lm >> 16) score(c0 + (lm & 0xFFFFu), lm >> 16, best);
                need = (int)best.need(na, cmin) - hcnt;
                low = weak(need, (float)sum, min((int64_t)A.kt, A.k - c0));
                if (low) {
                    if (t < 64) again |= 1ull << t;
                    else hard = true;
                }
            }
            if (low || need > (int)(lm >> 16)) {  // taken again, or above every counter
                for (int v = 0; v < nv; v++) c4[v * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
                __syncwarp();
                continue;
            }
            for (int v = 0; v < nv; v++) {
                const uint4 q = c4[v * 32 + lane];
                c4[v * 32 + lane] = make_uint4(0u, 0u, 0u, 0u);
                if (need > (int)C::TOP) continue;  // the bound rose above every counter
                const uint32_t ww[4] = {q.x, q.y, q.z, q.w};
                // a counter b <= TOP reaches `need` exactly when b + TOP - need sets its top bit
                const uint32_t add = (C::TOP - (uint32_t)need) * C::ONES, top = C::TOP * C::ONES;
                uint32_t hit[4];
#pragma unroll
                for (int u = 0; u < 4; u++) hit[u] = (ww[u] + add) & top;
                JxBest b = best;
                if (hit[0] | hit[1] | hit[2] | hit[3]) {
#pragma unroll
                    for (int u = 0; u < 4; u++)
                        for (uint32_t m = hit[u]; m; m &= m - 1) {
                            const int p = (__ffs((int)m) - 1) / C::CBITS;
                            score(c0 + ((((v * 32 + lane) * 4 + u) << C::LG) + p), (ww[u] >> (p * C::CBITS)) & C::CMASK, b);
                        }
                }
                if (__any_sync(0xffffffffu, b.j != best.j)) {
                    b.warp_merge();
                    best = b;
                    need = (int)best.need(na, cmin) - hcnt;  // does not fall: stays positive
                }
            }
            __syncwarp();
        }
        // no positive J: every fraction is 0 and the smallest index wins
        if (lane == 0) {
            if (hard) hard_rows[atomicAdd(n_hard, 1ull)] = make_int4((int)i, (int)best.n, (int)best.d, best.j);
            else A.labels[i] = best.n > 0 ? best.j : 0;
        }
    }
}

template <bool NARROW, int MW>  // MW: mask words per centre
__global__ void __launch_bounds__(JX_THREADS, 3) k_jac_count(JxArgs A, const uint64_t *__restrict__ cmask,
                                                             const int32_t *__restrict__ fq_list,
                                                             const int4 *__restrict__ rows,
                                                             const unsigned long long *__restrict__ n_rows) {
    using C = Jx<NARROW>;
    extern __shared__ uint4 jx_smem[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nv = A.kt / C::STEP;
    uint4 *c4 = jx_smem + (size_t)w * nv * 32;
    uint32_t *cw = reinterpret_cast<uint32_t *>(c4);
    int32_t *ridx = reinterpret_cast<int32_t *>(jx_smem + (size_t)JX_WARPS * nv * 32) + w * C::MAXI;
    for (int v = lane; v < nv * 32; v += 32) c4[v] = make_uint4(0u, 0u, 0u, 0u);
    const int64_t nwarps = (int64_t)gridDim.x * JX_WARPS, nr = (int64_t)*n_rows;
    for (int64_t q = (int64_t)blockIdx.x * JX_WARPS + w; q < nr; q += nwarps) {
        const int4 row = rows[q];  // the set and its best centre so far
        const int64_t i = row.x;
        const int64_t s0 = A.off[i];
        const int ni = (int)(A.off[i + 1] - s0);  // <= MAXI: the first pass listed it
        const uint32_t na = (uint32_t)(A.na_fix >= 0 ? A.na_fix : ni);
        uint64_t am[MW] = {};
        __syncwarp();
#pragma unroll 2
        for (int p = lane; p < ni; p += 32) {
            int32_t r = A.X.find(A.items[s0 + p]);
            if (r < -1) {
                const int hb = -2 - r;
#pragma unroll
                for (int h = 0; h < MW; h++)
                    if (hb >> 6 == h) am[h] |= 1ull << (hb & 63);
                r = fq_list[hb];
            }
            ridx[p] = r;
        }
        __syncwarp();
#pragma unroll
        for (int h = 0; h < MW; h++)
            am[h] = ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(am[h] >> 32)) << 32) |
                    __reduce_or_sync(0xffffffffu, (uint32_t)am[h]);
        JxBest best;
        best.n = (uint32_t)row.y;
        best.d = (uint32_t)row.z;
        best.j = row.w;
        for (int t = 0; t < A.ntiles; t++) {
            const int64_t c0 = (int64_t)t * A.kt;
            int sum = 0;
            jx_count<C>(cw, ridx, ni, t, A, sum);
            __syncwarp();
            const uint32_t need = best.need(na, (uint32_t)A.tile_min[t]);
            const int nc = (int)min((int64_t)A.kt, A.k - c0);
#pragma unroll 4
            for (int cc = lane; cc < nc; cc += 32) {
                uint32_t in = (cw[cc >> C::LG] >> ((cc & ((1 << C::LG) - 1)) * C::CBITS)) & C::CMASK;
#pragma unroll
                for (int h = 0; h < MW; h++) in += __popcll(am[h] & cmask[(c0 + cc) * MW + h]);
                if (in >= need) best.push(in, na + (uint32_t)A.clen[c0 + cc] - in, (int)(c0 + cc));
            }
            best.warp_merge();
            __syncwarp();
            for (int v = lane; v < nv * 32; v += 32) c4[v] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
        }
        if (lane == 0) A.labels[i] = best.n > 0 ? best.j : 0;
    }
}

// The same for narrow sets and one mask word, eight sets of a block scored together,
// thread per counter word: a centre's mask and size are loaded once for eight
// sets.  A warp of k_jac_count loads them for its one set, from L2 once the masks of
// k centres no longer fit the L1 beside the counters: 1.1M sets of 59 items, k = 6,993,
// 7.2 ms, here 5.4; 180,242 of 21, k = 10,817, 3.3 and 2.2; 2M of 59, k = 46,553, 23.0 and 21.5;
// where increments outweigh the scoring it is the other way, the warps of a block wait
// for one another: 300,000 of 59, k = 19,375, 5.5 and 5.8.
__global__ void __launch_bounds__(JX_THREADS, 3) k_jac_count8(JxArgs A, const uint64_t *__restrict__ cmask,
                                                              const int32_t *__restrict__ fq_list,
                                                              const int4 *__restrict__ rows,
                                                              const unsigned long long *__restrict__ n_rows) {
    using C = Jx<true>;
    constexpr int V = 1 << C::LG;  // counters of a word
    extern __shared__ uint4 jx_smem[];
    __shared__ int4 s_row[JX_WARPS];  // the sets and their best centres so far
    __shared__ uint64_t s_am[JX_WARPS];
    __shared__ uint32_t s_na[JX_WARPS];
    __shared__ uint32_t s_best[JX_WARPS][JX_WARPS][3];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int nv = A.kt / C::STEP;
    uint4 *c4 = jx_smem + (size_t)w * nv * 32;
    uint32_t *cw = reinterpret_cast<uint32_t *>(c4);
    const uint32_t *all = reinterpret_cast<const uint32_t *>(jx_smem);
    int32_t *ridx = reinterpret_cast<int32_t *>(jx_smem + (size_t)JX_WARPS * nv * 32) + w * C::MAXI;
    for (int v = lane; v < nv * 32; v += 32) c4[v] = make_uint4(0u, 0u, 0u, 0u);
    const int64_t nr = (int64_t)*n_rows;
    for (int64_t q0 = (int64_t)blockIdx.x * JX_WARPS; q0 < nr; q0 += (int64_t)gridDim.x * JX_WARPS) {
        const bool on = q0 + w < nr;
        const int4 row = on ? rows[q0 + w] : make_int4(-1, 0, 1, 0x7FFFFFFF);
        const int64_t s0 = on ? A.off[row.x] : 0;
        const int ni = on ? (int)(A.off[row.x + 1] - s0) : 0;  // <= MAXI: the first pass listed it
        uint64_t am = 0;
        for (int p = lane; p < ni; p += 32) {
            int32_t r = A.X.find(A.items[s0 + p]);
            if (r < -1) {
                const int hb = -2 - r;
                if (hb < 64) am |= 1ull << hb;
                r = fq_list[hb];
            }
            ridx[p] = r;
        }
        am = ((uint64_t)__reduce_or_sync(0xffffffffu, (uint32_t)(am >> 32)) << 32) |
             __reduce_or_sync(0xffffffffu, (uint32_t)am);
        if (lane == 0) {
            s_row[w] = row;
            s_am[w] = am;
            s_na[w] = (uint32_t)(A.na_fix >= 0 ? A.na_fix : ni);
        }
        __syncthreads();
        JxBest best[JX_WARPS];
        uint64_t ams[JX_WARPS];
        uint32_t na[JX_WARPS];
#pragma unroll
        for (int u = 0; u < JX_WARPS; u++) {
            best[u].n = (uint32_t)s_row[u].y;
            best[u].d = (uint32_t)s_row[u].z;
            best[u].j = s_row[u].w;
            ams[u] = s_am[u];
            na[u] = s_na[u];
        }
        for (int t = 0; t < A.ntiles; t++) {
            const int64_t c0 = (int64_t)t * A.kt;
            int sum = 0;
            jx_count<C>(cw, ridx, ni, t, A, sum);
            __syncthreads();
            const int nc = (int)min((int64_t)A.kt, A.k - c0);
            for (int x = threadIdx.x; x * V < nc; x += JX_THREADS) {
                // whole words: masks and sizes have room for the last one's
                uint64_t cm[V];
                int cl[V];
#pragma unroll
                for (int v = 0; v < V; v += 2) {
                    const ulonglong2 m2 = *reinterpret_cast<const ulonglong2 *>(cmask + c0 + x * V + v);
                    const int2 l2 = *reinterpret_cast<const int2 *>(A.clen + c0 + x * V + v);
                    cm[v] = m2.x;
                    cm[v + 1] = m2.y;
                    cl[v] = l2.x;
                    cl[v + 1] = l2.y;
                }
#pragma unroll
                for (int u = 0; u < JX_WARPS; u++) {
                    const uint32_t word = all[(size_t)u * nv * 128 + x];
#pragma unroll
                    for (int v = 0; v < V; v++) {
                        const uint32_t in = ((word >> (v * C::CBITS)) & C::CMASK) + (uint32_t)__popcll(ams[u] & cm[v]);
                        const uint32_t un = na[u] + (uint32_t)cl[v] - in;
                        if (in * best[u].d >= best[u].n * un && x * V + v < nc && in)
                            best[u].push(in, un, (int)(c0 + x * V + v));
                    }
                }
            }
            __syncthreads();
            for (int v = lane; v < nv * 32; v += 32) c4[v] = make_uint4(0u, 0u, 0u, 0u);
            __syncwarp();
        }
#pragma unroll
        for (int u = 0; u < JX_WARPS; u++) {
            best[u].warp_merge();
            if (lane == 0) {
                s_best[u][w][0] = best[u].n;
                s_best[u][w][1] = best[u].d;
                s_best[u][w][2] = (uint32_t)best[u].j;
            }
        }
        __syncthreads();
        if (on && lane == 0) {
            JxBest b;
            for (int u = 0; u < JX_WARPS; u++) b.push(s_best[w][u][0], s_best[w][u][1], (int)s_best[w][u][2]);
            A.labels[row.x] = b.n > 0 ? b.j : 0;
        }
    }
}

}  // namespace

// Majority set of each group of sets: items present in more than half of
// the group's member sets (groups CSR goff/gmem of set indices; sets CSR
// soff/sids).  Output CSR has one (possibly empty) entry per group.
geek_status majority_per_group(geek_ctx *ctx, Scratch &scr, int64_t ng, const int64_t *goff, const int32_t *gmem,
                               int64_t m, const int64_t *soff, const uint32_t *sids, int64_t **out_off,
                               uint32_t **out_ids, int64_t *out_n, cudaStream_t st) {
    int64_t *w, *woff, *T_dev, *cnt, *coff, *tot;
    int32_t *gid;
    GK_TRY(scr.alloc(&w, std::max<int64_t>(m, 1)));
    GK_TRY(scr.alloc(&woff, std::max<int64_t>(m, 1)));
    GK_TRY(scr.alloc(&gid, std::max<int64_t>(m, 1)));
    GK_TRY(scr.alloc(&T_dev, 1));
    GK_TRY(scr.alloc(&cnt, ng));
    GK_TRY(scr.alloc(out_off, ng + 1));
    GK_TRY(scr.alloc(&tot, 1));
    GK_CUDA(ctx, cudaMemsetAsync(cnt, 0, sizeof(int64_t) * ng, st));
    GK_COUNT();
    k_group_w<<<G(ctx, m), 256, 0, st>>>(m, gmem, soff, w);
    GK_COUNT();
    k_group_of<<<G(ctx, ng), 256, 0, st>>>(ng, goff, gid);
    GK_LAUNCH(ctx);
    GK_TRY(exclusive_scan_i64(ctx, scr, w, woff, m, T_dev, st));
    int64_t T = 0;
    GK_CUDA(ctx, cudaMemcpyAsync(&T, T_dev, 8, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    int64_t total = 0;
    if (T > 0) {
        uint64_t *pairs;
        GK_TRY(scr.alloc(&pairs, T));
        GK_COUNT();
        k_group_expand<<<G(ctx, m), 256, 0, st>>>(m, gid, gmem, woff, soff, sids, pairs);
        GK_LAUNCH(ctx);
        GK_TRY(radix_sort_segments(ctx, scr, 1, T, &pairs, nullptr, nullptr, 32 + bit_length_u64((uint64_t)ng), st));
        int64_t *prs, *nr;
        GK_TRY(scr.alloc(&prs, T + 1));
        GK_TRY(scr.alloc(&nr, 1));
        GK_TRY(segment_runs(ctx, scr, 1, T, pairs, nullptr, nullptr, prs, nr, st));
        int64_t NR = 0;
        GK_CUDA(ctx, cudaMemcpyAsync(&NR, nr, 8, cudaMemcpyDeviceToHost, st));
        GK_CUDA(ctx, cudaStreamSynchronize(st));
        int64_t *keep, *pos, *ktot;
        GK_TRY(scr.alloc(&keep, NR));
        GK_TRY(scr.alloc(&pos, NR));
        GK_TRY(scr.alloc(&ktot, 1));
        GK_COUNT();
        k_group_keep<<<G(ctx, NR), 256, 0, st>>>(nr, prs, pairs, goff, keep, cnt);
        GK_LAUNCH(ctx);
        GK_TRY(exclusive_scan_i64(ctx, scr, keep, pos, NR, ktot, st));
        GK_CUDA(ctx, cudaMemcpyAsync(&total, ktot, 8, cudaMemcpyDeviceToHost, st));
        GK_TRY(sort_err_check(ctx, st));  // synchronises st
        GK_TRY(scr.alloc(out_ids, std::max<int64_t>(1, total)));
        GK_COUNT();
        k_group_emit<<<G(ctx, NR), 256, 0, st>>>(nr, prs, pairs, keep, pos, *out_ids);
        GK_LAUNCH(ctx);
    } else {
        GK_TRY(scr.alloc(out_ids, 1));
    }
    GK_TRY(exclusive_scan_i64(ctx, scr, cnt, *out_off, ng, tot, st));
    GK_CUDA(ctx, cudaMemcpyAsync(*out_off + ng, tot, 8, cudaMemcpyDeviceToDevice, st));
    *out_n = total;
    (void)coff;
    return GEEK_OK;
}

geek_status assign_hetero(geek_ctx *ctx, Scratch &scr, const geek_buckets *b, const uint32_t *tok, int n_cat,
                          const silk_seeds *s, int32_t *labels, geek_assign_stats *stats, geek_centres *keep,
                          cudaStream_t st) {
    const int64_t n = b->n, k = s->k;
    const int A = b->L + n_cat;
    if (stats) *stats = geek_assign_stats{0.0, 0.0, k, 0};
    if (A > CAT_MAXA) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "more than %d categorical attributes", CAT_MAXA);
    if (n == 0) return GEEK_OK;
    uint64_t *attrs, *modes;
    GK_TRY(scr.alloc(&attrs, (size_t)n * A));
    GK_TRY(scr.alloc(&modes, (size_t)std::max<int64_t>(k, 1) * A));
    int32_t *rep = nullptr;
    if (keep && k) GK_TRY(scr.alloc(&rep, (size_t)k * A));
    GK_COUNT();
    k_build_attrs<<<G(ctx, n * A), 256, 0, st>>>(n, b->L, n_cat, b->num_key, tok, attrs);
    if (k) GK_COUNT(), k_modes<<<G(ctx, k * A), 256, 0, st>>>(k, A, s->off, s->ids, attrs, modes, rep);
    GK_LAUNCH(ctx);
    if (keep) {
        keep->kind = GEEK_HETERO;
        keep->k = k;
        keep->n_attr = A;
        GK_TRY(own_alloc(ctx, (void **)&keep->modes, sizeof(int64_t) * (size_t)std::max<int64_t>(k, 1) * A, st));
        if (k) {
            int64_t *flags, *excl, *tbase;
            GK_TRY(scr.alloc(&flags, std::max<int64_t>(b->NB, 1)));
            GK_TRY(scr.alloc(&excl, std::max<int64_t>(b->NB, 1)));
            GK_TRY(scr.alloc(&tbase, b->L));
            std::vector<int64_t> hb(b->L, 0);
            for (int l = 1; l < b->L; l++) hb[l] = hb[l - 1] + b->nb[l - 1];
            GK_CUDA(ctx, cudaMemcpyAsync(tbase, hb.data(), sizeof(int64_t) * b->L, cudaMemcpyHostToDevice, st));
            for (int l = 0; l < b->L; l++) {
                GK_COUNT();
                k_num_run_flags<<<G(ctx, b->nb[l]), 256, 0, st>>>(b->nb[l], hb[l], b->boff, b->members,
                                                                 b->num_key + (int64_t)l * n, flags);
            }
            GK_LAUNCH(ctx);
            GK_TRY(exclusive_scan_i64(ctx, scr, flags, excl, b->NB, nullptr, st));
            GK_COUNT();
            k_mode_out<<<G(ctx, k * A), 256, 0, st>>>(k, A, b->L, n, modes, rep, b->obj_bucket, tbase, excl, flags,
                                                      keep->modes);
            GK_LAUNCH(ctx);
            // the host vector hb must outlive the copy above
            GK_CUDA(ctx, cudaStreamSynchronize(st));
        }
    }
    unsigned long long *hist;  // rows by their number of matching attributes
    GK_TRY(scr.alloc(&hist, A + 1));
    GK_CUDA(ctx, cudaMemsetAsync(hist, 0, sizeof(unsigned long long) * (A + 1), st));
    bool done = false;
    if (match_bits_eligible(k, A))
        GK_TRY(match_bits_assign(ctx, scr, n, A, attrs, k, modes, labels, stats ? hist : nullptr, &done, st));
    if (!done) {
        GK_COUNT();
        k_assign_cat<<<(unsigned)ceil_div(n, 256), 256, 0, st>>>(n, A, k, attrs, modes, labels, stats ? hist : nullptr);
        GK_LAUNCH(ctx);
    }
    if (stats) {
        // the categorical distance 1 - m / (2A - m) takes A + 1 values: the
        // SSE is their sum weighted by the rows that have each
        unsigned long long hm[CAT_MAXA + 1];
        GK_CUDA(ctx, cudaMemcpyAsync(hm, hist, sizeof(unsigned long long) * (A + 1), cudaMemcpyDeviceToHost, st));
        GK_CUDA(ctx, cudaStreamSynchronize(st));
        double sse = 0.0, rmax = 0.0;
        for (int m = A; m >= 0; m--) {
            if (!hm[m]) continue;
            const double dd = 1.0 - (double)m / (double)(2 * A - m);
            sse += (double)hm[m] * dd;
            rmax = std::max(rmax, dd);
        }
        stats->sse = sse;
        stats->radius_max = rmax;
    }
    return GEEK_OK;
}

geek_status jaccard_core(geek_ctx *ctx, Scratch &scr, const int64_t *off, const uint32_t *items, int64_t n,
                         int na_fix, int64_t k, const int64_t *coff, const uint32_t *citems, int64_t nci,
                         int32_t *labels, geek_assign_stats *stats, cudaStream_t st);

geek_status assign_sets(geek_ctx *ctx, Scratch &scr, const int64_t *off, const uint32_t *items, int64_t n,
                        const silk_seeds *s, int32_t *labels, geek_assign_stats *stats, geek_centres *keep,
                        cudaStream_t st) {
    const int64_t k = s->k;
    if (stats) *stats = geek_assign_stats{0.0, 0.0, k, 0};
    if (keep) {
        keep->kind = GEEK_SETS;
        keep->k = k;
    }
    if (n == 0 || k == 0) {
        if (keep) {
            GK_TRY(own_alloc(ctx, (void **)&keep->item_off, sizeof(int64_t) * (size_t)(k + 1), st));
            GK_CUDA(ctx, cudaMemsetAsync(keep->item_off, 0, sizeof(int64_t) * (size_t)(k + 1), st));
        }
        if (n && k == 0) GK_CUDA(ctx, cudaMemsetAsync(labels, 0xFF, sizeof(int32_t) * n, st));
        return GEEK_OK;
    }
    // centres: majority item sets of the seeds
    int64_t *coff, nci = 0;
    uint32_t *citems;
    GK_TRY(majority_per_group(ctx, scr, k, s->off, s->ids, s->n_ids, off, items, &coff, &citems, &nci, st));
    if (keep) {
        keep->n_items = nci;
        GK_TRY(own_alloc(ctx, (void **)&keep->item_off, sizeof(int64_t) * (size_t)(k + 1), st));
        GK_TRY(own_alloc(ctx, (void **)&keep->items, sizeof(uint32_t) * (size_t)std::max<int64_t>(nci, 1), st));
        GK_CUDA(ctx, cudaMemcpyAsync(keep->item_off, coff, sizeof(int64_t) * (size_t)(k + 1), cudaMemcpyDeviceToDevice, st));
        if (nci)
            GK_CUDA(ctx, cudaMemcpyAsync(keep->items, citems, sizeof(uint32_t) * (size_t)nci, cudaMemcpyDeviceToDevice, st));
    }
    return jaccard_core(ctx, scr, off, items, n, -1, k, coff, citems, nci, labels, stats, st);
}

// Exact Jaccard argmax of every set against k centre sets (CSR coff /
// citems, nci items): J_j = |A n C_j| / |A u C_j|, larger fraction then
// smaller index; with no positive J the label is 0.  na_fix >= 0 gives every
// set the size na_fix (rows padded with an id that no centre holds).
geek_status jaccard_core(geek_ctx *ctx, Scratch &scr, const int64_t *off, const uint32_t *items, int64_t n,
                         int na_fix, int64_t k, const int64_t *coff, const uint32_t *citems, int64_t nci,
                         int32_t *labels, geek_assign_stats *stats, cudaStream_t st) {
    // inverted index item -> centres: pairs sorted by (item, centre), runs of
    // equal items, one posting list (ascending centres) per distinct item
    uint64_t *pairs, *ikey;
    GK_TRY(scr.alloc(&pairs, std::max<int64_t>(nci, 1)));
    GK_TRY(scr.alloc(&ikey, std::max<int64_t>(nci, 1)));
    GK_COUNT();
    k_centre_pairs<<<G(ctx, k), 256, 0, st>>>(k, coff, citems, pairs);
    GK_LAUNCH(ctx);
    GK_TRY(radix_sort_segments(ctx, scr, 1, nci, &pairs, nullptr, nullptr, 64, st));
    GK_COUNT();
    k_item_key<<<G(ctx, nci), 256, 0, st>>>(nci, pairs, ikey);
    GK_LAUNCH(ctx);
    int64_t *rs, *nr_dev;
    GK_TRY(scr.alloc(&rs, nci + 1));
    GK_TRY(scr.alloc(&nr_dev, 1));
    GK_TRY(segment_runs(ctx, scr, 1, nci, ikey, nullptr, nullptr, rs, nr_dev, st));
    int64_t ni = 0;
    GK_CUDA(ctx, cudaMemcpyAsync(&ni, nr_dev, 8, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    unsigned long long h_amax = 0, *d_amax;  // items of the largest set
    GK_TRY(scr.alloc(&d_amax, 1));
    GK_CUDA(ctx, cudaMemsetAsync(d_amax, 0, sizeof(unsigned long long), st));
    if (na_fix < 0 && n > 0) {
        GK_COUNT();
        k_max_len<<<G(ctx, n), 256, 0, st>>>(n, off, d_amax);
        GK_LAUNCH(ctx);
    }
    // heavy items: the (up to 64 JX_HW) longest posting lists of length >= 2,
    // chosen on the host from the run lengths; the others keep posting lists
    std::vector<int64_t> hrs(ni + 1);
    GK_CUDA(ctx, cudaMemcpyAsync(hrs.data(), rs, 8 * (ni + 1), cudaMemcpyDeviceToHost, st));
    std::vector<int32_t> ord(ni);
    GK_CUDA(ctx, cudaMemcpyAsync(&h_amax, d_amax, sizeof h_amax, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    // the narrow kernels when no set has more than their MAXI items
    const bool narrow = (na_fix >= 0 ? (int64_t)na_fix : (int64_t)h_amax) <= Jx<true>::MAXI;
    for (int64_t r = 0; r < ni; r++) ord[r] = (int32_t)r;
    const int64_t fmax = std::min<int64_t>(64 * JX_MW, ni);
    std::partial_sort(ord.begin(), ord.begin() + fmax, ord.end(), [&](int32_t a, int32_t b) {
        const int64_t la = hrs[a + 1] - hrs[a], lb = hrs[b + 1] - hrs[b];
        return la != lb ? la > lb : a < b;
    });
    int nfreq = 0;  // frequent items, by rank: the first nheavy of them are the heavy ones
    while (nfreq < fmax && hrs[ord[nfreq] + 1] - hrs[ord[nfreq]] >= 2) nfreq++;
    const int nheavy = std::min(nfreq, 64 * jx_heavy_words(hrs, ord, nfreq, k, narrow));
    const int HW = (nheavy + 63) / 64, FW = (nfreq + 63) / 64;
    std::vector<int32_t> fq_runs(ord.begin(), ord.begin() + nfreq);
    std::sort(fq_runs.begin(), fq_runs.end());
    std::vector<int16_t> f_bit(nfreq);
    std::vector<int64_t> h_is(ni, 0);
    std::vector<int32_t> hv_runs(ord.begin(), ord.begin() + nheavy);
    std::sort(hv_runs.begin(), hv_runs.end());  // runs ascend with the item value
    std::vector<int16_t> h_bit(nheavy);
    std::vector<int32_t> rank_of(ni, -1);
    for (int b = 0; b < nfreq; b++) rank_of[ord[b]] = b;  // bit = rank by posting length
    for (int q = 0; q < nfreq; q++) f_bit[q] = (int16_t)rank_of[fq_runs[q]];
    for (int q = 0; q < nheavy; q++) {
        h_is[hv_runs[q]] = 1;
        h_bit[q] = (int16_t)rank_of[hv_runs[q]];
    }
    uint32_t *d_litem, *d_lcentre, *hv_item;
    int16_t *hv_bit;
    int64_t *is_heavy, *lrun, *lrun_pos, *lent, *lent_pos, *d_loff, *nlight, *nlent, *hv_run_dev;
    GK_TRY(scr.alloc(&is_heavy, std::max<int64_t>(ni, 1)));
    GK_TRY(scr.alloc(&hv_item, std::max(1, nheavy)));
    GK_TRY(scr.alloc(&hv_bit, std::max(1, nheavy)));
    GK_TRY(scr.alloc(&hv_run_dev, std::max(1, nheavy)));
    GK_TRY(scr.alloc(&lrun, std::max<int64_t>(ni, 1)));
    GK_TRY(scr.alloc(&lrun_pos, std::max<int64_t>(ni, 1)));
    GK_TRY(scr.alloc(&lent, std::max<int64_t>(ni, 1)));
    GK_TRY(scr.alloc(&lent_pos, std::max<int64_t>(ni, 1)));
    GK_TRY(scr.alloc(&nlight, 1));
    GK_TRY(scr.alloc(&nlent, 1));
    uint32_t *fq_item;
    int16_t *fq_bit;
    int64_t *fq_run_dev;
    int32_t *fq_list;
    GK_TRY(scr.alloc(&fq_item, std::max(1, nfreq)));
    GK_TRY(scr.alloc(&fq_bit, std::max(1, nfreq)));
    GK_TRY(scr.alloc(&fq_run_dev, std::max(1, nfreq)));
    GK_TRY(scr.alloc(&fq_list, std::max(1, nfreq)));
    GK_CUDA(ctx, cudaMemcpyAsync(is_heavy, h_is.data(), 8 * ni, cudaMemcpyHostToDevice, st));
    if (nfreq) {
        std::vector<int64_t> fq_r64(fq_runs.begin(), fq_runs.end());
        GK_CUDA(ctx, cudaMemcpyAsync(fq_run_dev, fq_r64.data(), 8 * nfreq, cudaMemcpyHostToDevice, st));
        GK_CUDA(ctx, cudaMemcpyAsync(fq_bit, f_bit.data(), 2 * nfreq, cudaMemcpyHostToDevice, st));
        GK_COUNT();
        k_run_items<<<G(ctx, nfreq), 256, 0, st>>>(nfreq, fq_run_dev, rs, ikey, fq_item);
        GK_LAUNCH(ctx);
    }
    if (nheavy) {
        std::vector<int64_t> hv_r64(hv_runs.begin(), hv_runs.end());
        GK_CUDA(ctx, cudaMemcpyAsync(hv_run_dev, hv_r64.data(), 8 * nheavy, cudaMemcpyHostToDevice, st));
        GK_CUDA(ctx, cudaMemcpyAsync(hv_bit, h_bit.data(), 2 * nheavy, cudaMemcpyHostToDevice, st));
        GK_COUNT();
        k_run_items<<<G(ctx, nheavy), 256, 0, st>>>(nheavy, hv_run_dev, rs, ikey, hv_item);
        GK_LAUNCH(ctx);
    }
    // the host vectors above must outlive their copies
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    GK_COUNT();
    k_light_flags<<<G(ctx, ni), 256, 0, st>>>(ni, rs, is_heavy, lrun, lent);
    GK_LAUNCH(ctx);
    GK_TRY(exclusive_scan_i64(ctx, scr, lrun, lrun_pos, ni, nlight, st));
    GK_TRY(exclusive_scan_i64(ctx, scr, lent, lent_pos, ni, nlent, st));
    int64_t h_nlight = 0, h_nlent = 0;
    GK_CUDA(ctx, cudaMemcpyAsync(&h_nlight, nlight, 8, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaMemcpyAsync(&h_nlent, nlent, 8, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    GK_TRY(scr.alloc(&d_litem, std::max<int64_t>(1, h_nlight)));
    GK_TRY(scr.alloc(&d_loff, h_nlight + 1));
    GK_TRY(scr.alloc(&d_lcentre, std::max<int64_t>(1, h_nlent)));
    GK_COUNT();
    k_light_emit<<<G(ctx, ni), 256, 0, st>>>(ni, rs, ikey, pairs, is_heavy, lrun_pos, lent_pos, d_litem, d_loff,
                                             d_lcentre, nlent, h_nlight);
    GK_LAUNCH(ctx);
    if (nfreq) {
        GK_COUNT();
        k_freq_list<<<G(ctx, nfreq), 256, 0, st>>>(nfreq, nheavy, fq_run_dev, fq_bit, lrun_pos, fq_list);
        GK_LAUNCH(ctx);
    }
    uint64_t *cmask, *fmask;
    int32_t *clen, *counts;
    GK_TRY(scr.alloc(&cmask, (size_t)k * std::max(HW, 1) + 4));  // k_jac_count8 reads whole counter words
    GK_TRY(scr.alloc(&clen, k + 4));
    GK_COUNT();
    k_heavy_masks<JX_HW><<<G(ctx, k), 256, 0, st>>>(k, coff, citems, hv_item, hv_bit, nheavy, HW, cmask, clen);
    GK_TRY(scr.alloc(&fmask, (size_t)k * std::max(FW, 1)));
    GK_COUNT();
    k_heavy_masks<JX_MW><<<G(ctx, k), 256, 0, st>>>(k, coff, citems, fq_item, fq_bit, nfreq, FW, fmask, clen);
    GK_LAUNCH(ctx);
    if (nci > 0x7FFFFFFFLL) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "more than 2^31 centre items");
    // the tiled kernel compares fractions in 32 bits: |A| <= MAXI (else the
    // dense path) and every |C| below 2^15
    bool tiled_ok = na_fix < 32768;
    uint64_t h_last = 0;  // the largest item of any centre
    {
        std::vector<int64_t> hco(k + 1);
        GK_CUDA(ctx, cudaMemcpyAsync(hco.data(), coff, 8 * (k + 1), cudaMemcpyDeviceToHost, st));
        // the items ascend with the runs: the last entry holds the largest
        if (nci > 0)
            GK_CUDA(ctx, cudaMemcpyAsync(&h_last, ikey + nci - 1, sizeof h_last, cudaMemcpyDeviceToHost, st));
        GK_CUDA(ctx, cudaStreamSynchronize(st));
        for (int64_t j = 0; j < k && tiled_ok; j++) tiled_ok = hco[j + 1] - hco[j] < 32768;
    }
    int32_t *ovf;
    unsigned long long *n_ovf;
    GK_TRY(scr.alloc(&ovf, n));
    GK_TRY(scr.alloc(&n_ovf, 1));
    GK_CUDA(ctx, cudaMemsetAsync(n_ovf, 0, sizeof(unsigned long long), st));
    {
        // tiles of kt centres (the last one may be short), a multiple of the
        // counters one warp-wide load covers
        const int step = narrow ? Jx<true>::STEP : Jx<false>::STEP;
        const int kt = (int)std::min<int64_t>(narrow ? Jx<true>::KT : Jx<false>::KT, ceil_div(k, step) * step);
        const int ntiles = (int)ceil_div(k, kt);
        const size_t smem = (size_t)JX_WARPS * (narrow ? kt + 4 * Jx<true>::MAXI : 2 * kt + 4 * Jx<false>::MAXI);
        int32_t *toff, *tile_min;
        uint16_t *d_lloc;
        GK_TRY(scr.alloc(&toff, (size_t)std::max<int64_t>(h_nlight, 1) * (ntiles + 1)));
        GK_TRY(scr.alloc(&tile_min, ntiles));
        GK_TRY(scr.alloc(&d_lloc, std::max<int64_t>(1, h_nlent)));
        GK_COUNT();
        k_tile_offsets<<<G(ctx, h_nlight * (ntiles + 1)), 256, 0, st>>>(h_nlight, d_loff, d_lcentre, ntiles, kt, toff);
        GK_COUNT();
        k_tile_local<<<G(ctx, h_nlent), 256, 0, st>>>(h_nlent, d_lcentre, kt, d_lloc);
        GK_COUNT();
        k_tile_min_len<<<ntiles, 256, 0, st>>>(k, kt, clen, tile_min);
        // the largest centre item decides between the table and the searches:
        // above 2^24 (a 64 MB table) the fill would outweigh the searches' 20
        // dependent loads per item
        JxIndex X{nullptr, 0, fq_item, fq_bit, nfreq, d_litem, h_nlight};
        if (h_last < (1u << 24)) {
            int32_t *lut;
            X.n_lut = (int64_t)h_last + 1;
            GK_TRY(scr.alloc(&lut, (size_t)X.n_lut));
            GK_CUDA(ctx, cudaMemsetAsync(lut, 0xFF, sizeof(int32_t) * (size_t)X.n_lut, st));
            GK_COUNT();
            k_item_lut<<<G(ctx, h_nlight), 256, 0, st>>>(h_nlight, d_litem, lut);
            if (nfreq) {
                GK_COUNT();
                k_freq_lut<<<G(ctx, nfreq), 256, 0, st>>>(nfreq, fq_item, fq_bit, lut);
            }
            X.lut = lut;
        }
        EvTimer tk(ctx, "kernel.jaccard", st);
        tk.work = (double)n * (double)k;  // (set, centre) pairs decided
        if (!tiled_ok) {  // very large central sets: every set takes the dense path
            GK_COUNT();
            k_iota_rows<<<G(ctx, n), 256, 0, st>>>(n, ovf, n_ovf);
            GK_LAUNCH(ctx);
        } else {
        int4 *hard;
        unsigned long long *n_hard;
        GK_TRY(scr.alloc(&hard, n));
        GK_TRY(scr.alloc(&n_hard, 1));
        GK_CUDA(ctx, cudaMemsetAsync(n_hard, 0, sizeof(unsigned long long), st));
        const JxArgs A{n, off, items, na_fix, k, kt, ntiles, clen, tile_min, toff, d_lloc, X, labels};
        auto run = [&](auto *prune, auto *count) -> geek_status {
            int per_sm[2] = {1, 1};
            const void *fn[2] = {(const void *)prune, (const void *)count};
            for (int f = 0; f < 2; f++) {
                GK_CUDA(ctx, cudaFuncSetAttribute(fn[f], cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
                GK_CUDA(ctx, cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm[f], fn[f], JX_THREADS, smem));
            }
            auto grid = [&](int f) {
                return (unsigned)std::min<int64_t>(ceil_div(n, JX_WARPS), (int64_t)ctx->num_sms * std::max(per_sm[f], 1));
            };
            GK_COUNT();
            prune<<<grid(0), JX_THREADS, smem, st>>>(A, fmask, FW, ovf, n_ovf, hard, n_hard);
            GK_COUNT();
            count<<<grid(1), JX_THREADS, smem, st>>>(A, cmask, fq_list, hard, n_hard);
            GK_LAUNCH(ctx);
            return GEEK_OK;
        };
        if (narrow)
            GK_TRY(run(k_jac_prune<true>, HW > 2           ? k_jac_count<true, 3>
                                          : HW > 1         ? k_jac_count<true, 2>
                                          : k >= JX_BLOCKS ? k_jac_count8
                                                           : k_jac_count<true, 1>));
        else GK_TRY(run(k_jac_prune<false>, k_jac_count<false, 1>));
        GK_LAUNCH(ctx);
        }
    }
    unsigned long long h_ovf = 0;
    GK_CUDA(ctx, cudaMemcpyAsync(&h_ovf, n_ovf, sizeof h_ovf, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    if (h_ovf) {
        // sets with too many light candidates: every centre scanned per set
        const int blocks = (int)std::min<int64_t>(ctx->num_sms * 4, ceil_div((int64_t)h_ovf, 8));
        const int64_t nwarps = (int64_t)blocks * 8;
        GK_TRY(scr.alloc(&counts, (size_t)nwarps * k));
        GK_CUDA(ctx, cudaMemsetAsync(counts, 0, sizeof(int32_t) * nwarps * k, st));
        GK_COUNT();
        auto *dense = HW > 2 ? k_assign_jaccard<3> : HW > 1 ? k_assign_jaccard<2> : k_assign_jaccard<1>;
        dense<<<blocks, 256, 0, st>>>(n, off, items, k, clen, cmask, hv_item, hv_bit, nheavy, d_litem, d_loff, h_nlight,
                                      d_lcentre, counts, labels, ovf, n_ovf, na_fix);
        GK_LAUNCH(ctx);
    }
    if (stats) stats->n_recheck_rows = (int64_t)h_ovf;  // sets decided by the dense path
    return sort_err_check(ctx, st);  // synchronises st
}

namespace {

// id of each token in the sorted distinct list U (nu entries), or 2^32 - 1
// when absent (no centre holds it)
__global__ void k_map_tokens(int64_t m, const uint64_t *__restrict__ tok, const uint64_t *__restrict__ U, int64_t nu,
                             uint32_t *__restrict__ out) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t v = tok[e];
        int64_t lo = 0, hi = nu;
        while (lo < hi) {
            const int64_t mid = (lo + hi) >> 1;
            if (U[mid] < v) lo = mid + 1;
            else hi = mid;
        }
        out[e] = (lo < nu && U[lo] == v) ? (uint32_t)lo : 0xFFFFFFFFu;
    }
}

__global__ void k_fixed_off(int64_t n, int64_t len, int64_t *__restrict__ off) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i <= n; i += (int64_t)gridDim.x * blockDim.x)
        off[i] = i * len;
}

// the first token of each run of equal sorted tokens: compacted to U
__global__ void k_run_firsts(int64_t m, const uint64_t *__restrict__ sorted, const int64_t *__restrict__ rank_excl,
                             uint64_t *__restrict__ U) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        if (e == 0 || sorted[e] != sorted[e - 1]) U[rank_excl[e]] = sorted[e];
}

__global__ void k_run_flags(int64_t m, const uint64_t *__restrict__ sorted, int64_t *__restrict__ flags) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < m; e += (int64_t)gridDim.x * blockDim.x)
        flags[e] = (e == 0 || sorted[e] != sorted[e - 1]) ? 1 : 0;
}

}  // namespace

// Sparse sets reduced by DOPH (Alg. 3): every object is its D' tokens, one per
// reduced dimension.  Central vector = the mode of each dimension over the
// seed's members (Sect. 3.3: the mode of sparse data after DOPH; ties to the
// smallest token); distance 1 - Jaccard of the token sets, i.e. the label
// maximises the number of dimensions equal to the centre's mode
// (match_bits.cu).  Where the mask table would be too large, or has no room,
// tokens map to 32-bit ids of the distinct mode tokens and the Jaccard engine decides, with
// |A| = |C| = D'.
geek_status assign_doph(geek_ctx *ctx, Scratch &scr, const geek_buckets *b, const silk_seeds *s, int32_t *labels,
                        geek_assign_stats *stats, geek_centres *keep, cudaStream_t st) {
    const int64_t n = b->n, k = s->k;
    const int D = b->doph_bins;
    if (stats) *stats = geek_assign_stats{0.0, 0.0, k, 0};
    if (keep) {
        keep->kind = GEEK_SETS;
        keep->k = k;
        keep->n_attr = D;
        GK_TRY(own_alloc(ctx, (void **)&keep->modes, sizeof(int64_t) * (size_t)std::max<int64_t>(k, 1) * D, st));
    }
    if (n == 0) return GEEK_OK;
    if (k == 0) {
        GK_CUDA(ctx, cudaMemsetAsync(labels, 0xFF, sizeof(int32_t) * n, st));
        return GEEK_OK;
    }
    const int64_t km = k * D;
    uint64_t *modes, *srt;
    GK_TRY(scr.alloc(&modes, km));
    GK_TRY(scr.alloc(&srt, km));
    GK_COUNT();
    k_modes<<<G(ctx, km), 256, 0, st>>>(k, D, s->off, s->ids, b->doph_tok, modes, nullptr);
    GK_LAUNCH(ctx);
    if (keep) GK_CUDA(ctx, cudaMemcpyAsync(keep->modes, modes, 8 * km, cudaMemcpyDeviceToDevice, st));
    bool done = false;
    if (match_bits_eligible(k, D))
        GK_TRY(match_bits_assign(ctx, scr, n, D, b->doph_tok, k, modes, labels, nullptr, &done, st));
    if (done) return GEEK_OK;
    // distinct mode tokens, ascending
    GK_CUDA(ctx, cudaMemcpyAsync(srt, modes, 8 * km, cudaMemcpyDeviceToDevice, st));
    GK_TRY(radix_sort_segments(ctx, scr, 1, km, &srt, nullptr, nullptr, 64, st));
    int64_t *flags, *rexcl, *nu_dev;
    GK_TRY(scr.alloc(&flags, km));
    GK_TRY(scr.alloc(&rexcl, km));
    GK_TRY(scr.alloc(&nu_dev, 1));
    GK_COUNT();
    k_run_flags<<<G(ctx, km), 256, 0, st>>>(km, srt, flags);
    GK_LAUNCH(ctx);
    GK_TRY(exclusive_scan_i64(ctx, scr, flags, rexcl, km, nu_dev, st));
    int64_t nu = 0;
    GK_CUDA(ctx, cudaMemcpyAsync(&nu, nu_dev, 8, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    if (nu >= 0xFFFFFFFFLL) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "too many distinct mode tokens");
    uint64_t *U;
    GK_TRY(scr.alloc(&U, nu));
    GK_COUNT();
    k_run_firsts<<<G(ctx, km), 256, 0, st>>>(km, srt, rexcl, U);
    // centres and rows as id lists of fixed length D
    uint32_t *cid, *rid;
    int64_t *coff, *roff;
    GK_TRY(scr.alloc(&cid, km));
    GK_TRY(scr.alloc(&rid, n * D));
    GK_TRY(scr.alloc(&coff, k + 1));
    GK_TRY(scr.alloc(&roff, n + 1));
    GK_COUNT();
    k_map_tokens<<<G(ctx, km), 256, 0, st>>>(km, modes, U, nu, cid);
    GK_COUNT();
    k_map_tokens<<<G(ctx, n * D), 256, 0, st>>>(n * D, b->doph_tok, U, nu, rid);
    GK_COUNT();
    k_fixed_off<<<G(ctx, k + 1), 256, 0, st>>>(k, D, coff);
    GK_COUNT();
    k_fixed_off<<<G(ctx, n + 1), 256, 0, st>>>(n, D, roff);
    GK_LAUNCH(ctx);
    return jaccard_core(ctx, scr, roff, rid, n, D, k, coff, cid, km, labels, stats, st);
}
