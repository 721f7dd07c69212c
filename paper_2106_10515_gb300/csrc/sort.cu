// Device radix sort, run detection and prefix sums: the grouping machinery
// behind bucket formation (T[G(x)].push(j) in Algs. 2-3), SILK bins (Alg. 4)
// and majority voting.  Sorting is a stable LSD radix sort with 8-bit digits
// over S equal-length segments at once (one segment per hash table), so the
// L tables of a transform share every launch; each pass is one kernel whose
// tiles find their output offsets by decoupled look-back.
#include <cstdarg>

#include "common.cuh"

namespace {

constexpr int RS_THREADS = 256;
constexpr int RS_ITEMS = 10;
constexpr int RS_TILE = RS_THREADS * RS_ITEMS;  // 2560 elements per tile
constexpr int NWARP = RS_THREADS / 32;

// ---- block-wide exclusive scan helper (uint32, 1024 threads max) ----------
template <int NT>
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t *total, uint32_t *wsum) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    uint32_t x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) wsum[warp] = x;
    __syncthreads();
    if (warp == 0) {
        uint32_t s = lane < NT / 32 ? wsum[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            uint32_t y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o) s += y;
        }
        if (lane < NT / 32) wsum[lane] = s;  // inclusive warp totals
    }
    __syncthreads();
    uint32_t before = warp ? wsum[warp - 1] : 0;
    *total = wsum[NT / 32 - 1];
    __syncthreads();
    return before + x - v;
}

// exclusive scan in place of each segment's `len` counters; optional total
__global__ void __launch_bounds__(1024) k_seg_scan_u32(uint32_t *__restrict__ c, int64_t len,
                                                       int64_t *__restrict__ totals) {
    __shared__ uint32_t wsum[32];
    uint32_t *a = c + (int64_t)blockIdx.x * len;
    uint32_t carry = 0;
    for (int64_t base = 0; base < len; base += 1024 * 4) {
        int64_t p0 = base + (int64_t)threadIdx.x * 4;
        uint32_t v[4], s = 0;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            v[k] = p0 + k < len ? a[p0 + k] : 0u;
            s += v[k];
        }
        uint32_t tot;
        uint32_t ex = block_excl_scan<1024>(s, &tot, wsum) + carry;
#pragma unroll
        for (int k = 0; k < 4; k++) {
            if (p0 + k < len) a[p0 + k] = ex;
            ex += v[k];
        }
        carry += tot;
    }
    if (totals && threadIdx.x == 0) totals[blockIdx.x] = carry;
}

// ---- one-sweep passes (decoupled look-back) --------------------------------
// Digit totals do not change from one LSD pass to the next (a pass only
// permutes a segment), so one read of the keys gives every pass its global
// digit offsets.  Each pass is then a single kernel: a block takes the next
// tile of its segment in launch order (a global ticket), publishes the
// tile's per-digit count, and adds up its predecessors' counts by looking
// back through their published words until one carries an inclusive prefix.
// Word layout: bits 31..30 = state (0 empty, 1 tile count, 2 inclusive
// prefix), bits 29..0 = count; segments are limited to 2^30 - 1 elements.
constexpr uint32_t LB_AGG = 1u << 30, LB_PREFIX = 2u << 30, LB_MASK = (1u << 30) - 1;
constexpr int HIST_BLOCKS_PER_SEG = 96;

__device__ __forceinline__ unsigned long long sort_gtimer() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

// counts[seg][pass][256] += digit counts of every pass (counts zeroed first).
// Shared histograms per warp pair keep same-address atomics rare when a
// high digit takes few values.
__global__ void __launch_bounds__(256) k_rs_hist_all(const uint64_t *__restrict__ lo, const uint64_t *__restrict__ hi,
                                                     int64_t m, int bit0, int npass, uint32_t *__restrict__ counts) {
    extern __shared__ uint32_t hs[];  // [4][npass][256]
    const int seg = blockIdx.y, t = threadIdx.x, sub = (t >> 6);
    for (int i = t; i < 4 * npass * 256; i += 256) hs[i] = 0;
    __syncthreads();
    const uint64_t *l = lo + (int64_t)seg * m;
    const uint64_t *h = hi ? hi + (int64_t)seg * m : nullptr;
    uint32_t *my = hs + sub * npass * 256;
    for (int64_t p = (int64_t)blockIdx.x * 256 + t; p < m; p += (int64_t)gridDim.x * 256) {
        const uint64_t kl = l[p];
        const uint64_t kh = h ? h[p] : 0;
        for (int q = 0; q < npass; q++) {
            const int sh = bit0 + q * 8;
            const uint32_t d = (uint32_t)(((sh >= 64 ? kh : kl) >> (sh & 63)) & 0xFFu);
            atomicAdd(&my[q * 256 + d], 1u);
        }
    }
    __syncthreads();
    for (int i = t; i < npass * 256; i += 256) {
        const uint32_t c = hs[i] + hs[npass * 256 + i] + hs[2 * npass * 256 + i] + hs[3 * npass * 256 + i];
        if (c) atomicAdd(&counts[(int64_t)seg * npass * 256 + i], c);
    }
}

// exclusive scan of every (segment, pass) row of 256 digit counts, in place
__global__ void __launch_bounds__(256) k_rs_base_all(uint32_t *__restrict__ counts) {
    __shared__ uint32_t wsum[32];
    uint32_t *a = counts + (int64_t)blockIdx.x * 256;
    const uint32_t v = a[threadIdx.x];
    uint32_t tot;
    a[threadIdx.x] = block_excl_scan<256>(v, &tot, wsum);
}

// One pass.  A tile of RS_TILE elements is split into 8 warp slices; warp w
// reads its slice striped (item i of lane l is element w*IT*32 + i*32 + l),
// so (warp, item, lane) is input order.  Each warp ranks its elements per
// digit with match-any, the block turns per-warp counts into tile offsets,
// stages the tile in shared memory in (digit, input order) and writes it out
// contiguously per digit: coalesced, stable.  Small tiles and 4 blocks per
// SM: the pass is latency bound, and occupancy pays more than long tiles (16
// tables of 2M elements, 215 us a pass, half of HBM; tiles of 5,120 elements by
// 512 threads 237, by 1,024 threads 365; the next tile's loads in flight during the
// writes 222).
template <bool HI, bool VALS>
__global__ void __launch_bounds__(RS_THREADS, 4)
    k_rs_onesweep(const uint64_t *__restrict__ lo_in, const uint64_t *__restrict__ hi_in,
                  const uint32_t *__restrict__ v_in, uint64_t *__restrict__ lo_out,
                  uint64_t *__restrict__ hi_out, uint32_t *__restrict__ v_out, int64_t m, int tiles,
                  int dsel, int sh, const uint32_t *__restrict__ dbase, int dstride, uint32_t *__restrict__ look,
                  uint32_t *__restrict__ ticket, int *__restrict__ err, unsigned long long wait_ns,
                  int stall_tile) {
    __shared__ uint32_t whist[NWARP][256];
    __shared__ uint32_t tstart[256];
    __shared__ uint32_t gbase[256];
    __shared__ uint32_t wsum[32];
    __shared__ uint32_t s_idx;
    extern __shared__ uint64_t stage[];
    uint64_t *st_lo = stage;
    uint64_t *st_hi = stage + RS_TILE;
    uint32_t *st_v = (uint32_t *)(stage + (HI ? 2 : 1) * RS_TILE);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    if (t == 0) s_idx = atomicAdd(ticket, 1u);
#pragma unroll
    for (int w = 0; w < NWARP; w++) whist[w][t] = 0;
    __syncthreads();
    const uint32_t idx = s_idx;
    // tickets interleave the segments: a tile's predecessor in its own
    // segment took its ticket S tickets earlier
    const int S = (int)(gridDim.x / (uint32_t)tiles);
    const int seg = (int)(idx % (uint32_t)S), tile = (int)(idx / (uint32_t)S);
    const int64_t so = (int64_t)seg * m;
    const int64_t t0 = (int64_t)tile * RS_TILE;
    const uint32_t lt = (1u << lane) - 1;
    constexpr int IT = RS_TILE / RS_THREADS;
    uint64_t klo[IT], khi[IT];
    uint32_t vv[IT], dr[IT];
    // every load of the tile in flight before the first (synchronising) rank step
#pragma unroll
    for (int i = 0; i < IT; i++) {
        const int64_t p = t0 + warp * (IT * 32) + i * 32 + lane;
        const bool valid = p < m;
        klo[i] = valid ? lo_in[so + p] : 0;
        khi[i] = (HI && valid) ? hi_in[so + p] : 0;
        vv[i] = (VALS && valid) ? (v_in ? v_in[so + p] : (uint32_t)p) : 0;
    }
#pragma unroll
    for (int i = 0; i < IT; i++) {
        const bool valid = t0 + warp * (IT * 32) + i * 32 + lane < m;
        const uint32_t d = valid ? (uint32_t)(((dsel ? khi[i] : klo[i]) >> sh) & 0xFFu) : 256u;
        const uint32_t peers = __match_any_sync(0xffffffffu, d);
        const int leader = __ffs(peers) - 1;
        uint32_t old = 0;
        if (lane == leader && d < 256) {
            old = whist[warp][d];
            whist[warp][d] = old + __popc(peers);
        }
        old = __shfl_sync(0xffffffffu, old, leader);
        dr[i] = d | ((old + __popc(peers & lt)) << 9);
    }
    __syncthreads();
    uint32_t run = 0;
#pragma unroll
    for (int w = 0; w < NWARP; w++) {
        const uint32_t c = whist[w][t];
        whist[w][t] = run;
        run += c;
    }
    // publish this tile's count of digit t; the look-back comes after the
    // tile is staged, so that predecessors have had time to finish theirs
    uint32_t *lk = look + (int64_t)seg * tiles * 256;
    volatile uint32_t *vlk = lk;
    if (tile != stall_tile) vlk[(int64_t)tile * 256 + t] = (tile == 0 ? LB_PREFIX : LB_AGG) | run;
    uint32_t tot;
    tstart[t] = block_excl_scan<RS_THREADS>(run, &tot, wsum);
    __syncthreads();
#pragma unroll
    for (int i = 0; i < IT; i++) {
        const uint32_t d = dr[i] & 511u;
        if (d < 256) {
            const uint32_t lp = tstart[d] + whist[warp][d] + (dr[i] >> 9);
            st_lo[lp] = klo[i];
            if (HI) st_hi[lp] = khi[i];
            if (VALS) st_v[lp] = vv[i];
        }
    }
    // look back over the predecessors of this segment, four words per read
    uint32_t excl = 0;
    bool gave_up = false;
    if (tile > 0) {
        int j = tile - 1;
        unsigned long long w0 = 0;
        for (uint32_t it = 0;; it++) {
            uint32_t w[4];
#pragma unroll
            for (int k = 0; k < 4; k++) w[k] = j - k >= 0 ? vlk[(int64_t)(j - k) * 256 + t] : 0u;
            int k = 0;
            bool done = false;
            for (; k < 4; k++) {
                const uint32_t stt = w[k] & ~LB_MASK;
                if (stt == 0) break;  // not published yet: poll again from here
                excl += w[k] & LB_MASK;
                if (stt == LB_PREFIX) {
                    done = true;
                    break;
                }
            }
            if (done) break;
            j -= k;  // tile 0 always publishes a prefix, so j stays >= 0
            if (k == 0 && (it & 63) == 63) {
                const unsigned long long tn = sort_gtimer();
                if (w0 == 0) {
                    w0 = tn;
                } else if (tn - w0 > wait_ns) {
                    gave_up = true;
                    break;
                }
            }
        }
    }
    // A wait that ran out: the block recounts every digit of its
    // predecessors straight from this pass's input (a permutation of the
    // keys, so the counts are exact), which keeps the pass correct and every
    // write inside the segment; the call still reports GEEK_ERR_TIMEOUT.
    if (__syncthreads_or(gave_up)) {
        if (t == 0) atomicExch(err, (int)GEEK_ERR_TIMEOUT);
        gbase[t] = 0;
        __syncthreads();
        const uint64_t *src = dsel ? hi_in : lo_in;
        for (int64_t p = t; p < t0; p += RS_THREADS) atomicAdd(&gbase[(uint32_t)((src[so + p] >> sh) & 0xFFu)], 1u);
        __syncthreads();
        excl = gbase[t];
        __syncthreads();
    }
    if (tile > 0 && tile != stall_tile) vlk[(int64_t)tile * 256 + t] = LB_PREFIX | ((excl + run) & LB_MASK);
    // output position of staged element q of digit d: goff[d] + q
    gbase[t] = dbase[(int64_t)seg * dstride + t] + excl - tstart[t];
    __syncthreads();
    const int cnt = (int)min((int64_t)RS_TILE, m - t0);
    for (int q = t; q < cnt; q += RS_THREADS) {
        const uint64_t kl = st_lo[q];
        const uint64_t kh = HI ? st_hi[q] : 0;
        const uint32_t d = (uint32_t)(((dsel ? kh : kl) >> sh) & 0xFFu);
        const int64_t dst = so + (uint32_t)(gbase[d] + (uint32_t)q);
        lo_out[dst] = kl;
        if (HI) hi_out[dst] = kh;
        if (VALS) v_out[dst] = st_v[q];
    }
}

// Segments of at most RB_MAX elements: one block sorts a segment in shared
// memory, all passes in one launch (each pass of the tiled form is a launch of
// its own plus the digit totals: 19 launches for 64 bits).  Ranking as in
// k_rs_onesweep, the tile read back after each pass.  RB_MAX is what a thread's
// registers hold, 10 elements; a pass over it takes some 2 us, where a launch of
// the tiled form takes 3 to 7 for so few (the 20,000 x 32 pipeline, whose SILK
// tables are below the line: 1.85 -> 1.78 ms).
constexpr int RB_THREADS = 512, RB_ITEMS = 10, RB_MAX = RB_THREADS * RB_ITEMS, RB_WARPS = RB_THREADS / 32;
template <bool HI, bool VALS>
__global__ void __launch_bounds__(RB_THREADS) k_rs_block(uint64_t *__restrict__ lo, uint64_t *__restrict__ hi,
                                                         uint32_t *__restrict__ v, int m, int bit0, int npass, bool iota) {
    __shared__ uint32_t whist[RB_WARPS][256];
    __shared__ uint32_t tstart[256];
    __shared__ uint32_t wsum[32];
    extern __shared__ uint64_t stage[];
    uint64_t *st_lo = stage, *st_hi = stage + m;
    uint32_t *st_v = reinterpret_cast<uint32_t *>(stage + (HI ? 2 : 1) * (size_t)m);
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const int64_t so = (int64_t)blockIdx.x * m;
    const uint32_t lt = (1u << lane) - 1;
    uint64_t klo[RB_ITEMS], khi[RB_ITEMS];
    uint32_t vv[RB_ITEMS], dr[RB_ITEMS];
    const int p0 = warp * (RB_ITEMS * 32) + lane;
#pragma unroll
    for (int i = 0; i < RB_ITEMS; i++) {
        const int p = p0 + i * 32;
        klo[i] = p < m ? lo[so + p] : 0;
        khi[i] = HI && p < m ? hi[so + p] : 0;
        vv[i] = VALS && p < m ? (iota ? (uint32_t)p : v[so + p]) : 0;
    }
    for (int q = 0; q < npass; q++) {
        const int sh = bit0 + 8 * q;
        for (int e = t; e < RB_WARPS * 256; e += RB_THREADS) whist[e >> 8][e & 255] = 0;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RB_ITEMS; i++) {
            const uint32_t d = p0 + i * 32 < m ? (uint32_t)(((sh >= 64 ? khi[i] : klo[i]) >> (sh & 63)) & 0xFFu) : 256u;
            const uint32_t peers = __match_any_sync(0xffffffffu, d);
            const int leader = __ffs(peers) - 1;
            uint32_t old = 0;
            if (lane == leader && d < 256) {
                old = whist[warp][d];
                whist[warp][d] = old + __popc(peers);
            }
            old = __shfl_sync(0xffffffffu, old, leader);
            dr[i] = d | ((old + __popc(peers & lt)) << 9);
        }
        __syncthreads();
        uint32_t run = 0;
        if (t < 256) {
#pragma unroll
            for (int w = 0; w < RB_WARPS; w++) {
                const uint32_t c = whist[w][t];
                whist[w][t] = run;
                run += c;
            }
        }
        uint32_t tot;
        const uint32_t ex = block_excl_scan<RB_THREADS>(run, &tot, wsum);
        if (t < 256) tstart[t] = ex;
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RB_ITEMS; i++) {
            const uint32_t d = dr[i] & 511u;
            if (d < 256) {
                const uint32_t lp = tstart[d] + whist[warp][d] + (dr[i] >> 9);
                st_lo[lp] = klo[i];
                if (HI) st_hi[lp] = khi[i];
                if (VALS) st_v[lp] = vv[i];
            }
        }
        __syncthreads();
#pragma unroll
        for (int i = 0; i < RB_ITEMS; i++) {
            const int p = p0 + i * 32;
            if (p < m) {
                klo[i] = st_lo[p];
                if (HI) khi[i] = st_hi[p];
                if (VALS) vv[i] = st_v[p];
            }
        }
        // the next pass writes the stage only after its first barriers
    }
#pragma unroll
    for (int i = 0; i < RB_ITEMS; i++) {
        const int p = p0 + i * 32;
        if (p < m) {
            lo[so + p] = klo[i];
            if (HI) hi[so + p] = khi[i];
            if (VALS) v[so + p] = vv[i];
        }
    }
}

// ---- keys sorted by their upper bits, then settled ---------------------------
// m objects rarely need all the bits of a wide key to be told apart.  So the
// passes cover the upper bits only, and the runs of equal prefixes are put in the
// order of the whole key afterwards: short ones by one thread each, longer ones by
// a block each.  Both keep equal keys in the order they have, so the result is
// the full sort's.  How many passes leave few prefixes that repeat is estimated
// from a sample first (k_rs_twins).
constexpr int FX_RUN = 32;                        // longest run of one thread
constexpr int TW_SAMPLES = 8192, TW_SLOTS = 2 * TW_SAMPLES, TW_WIDTHS = 8;

__device__ __forceinline__ bool same_prefix(uint64_t l0, uint64_t h0, uint64_t l1, uint64_t h1, int bit0) {
    if (bit0 >= 64) return ((h0 ^ h1) >> (bit0 - 64)) == 0;
    return h0 == h1 && ((l0 ^ l1) >> bit0) == 0;
}

// twins[w] += the samples of every segment whose prefix above bit0 - 8 w another
// sample has, most[w] = the most samples of one prefix (block per segment and w;
// pseudo-random positions, so that any order of the objects is sampled alike; the
// multipliers are those of Knuth's multiplicative hash, the MurmurHash3 finalizer,
// degski's 64-bit mixer and SplitMix64's increment)
__global__ void __launch_bounds__(1024) k_rs_twins(const uint64_t *__restrict__ lo, const uint64_t *__restrict__ hi,
                                                   int64_t m, int bit0, unsigned long long *__restrict__ twins,
                                                   unsigned long long *__restrict__ most) {
    extern __shared__ unsigned long long slot[];
    uint32_t *const more = reinterpret_cast<uint32_t *>(slot + TW_SLOTS);  // samples after a slot's first
    const int64_t so = (int64_t)blockIdx.x * m;
    bit0 -= 8 * blockIdx.y;
    for (int e = threadIdx.x; e < TW_SLOTS; e += 1024) {
        slot[e] = ~0ull;
        more[e] = 0;
    }
    __syncthreads();
    unsigned found = 0, same = 0;
    for (int e = threadIdx.x; e < TW_SAMPLES; e += 1024) {
        // one position in each of TW_SAMPLES equal stretches
        uint32_t z = (uint32_t)e * 2654435761u + blockIdx.x * 0x9E3779B9u;
        z = (z ^ (z >> 15)) * 0x85EBCA6Bu;
        z = (z ^ (z >> 13)) * 0xC2B2AE35u;
        z ^= z >> 16;
        const int64_t a = e * m / TW_SAMPLES, b = (e + 1) * m / TW_SAMPLES;
        const int64_t p = so + a + (int64_t)(z % (uint32_t)(b - a));
        const uint64_t l = lo[p], h = hi[p];
        unsigned long long q = bit0 >= 64 ? h >> (bit0 - 64) : (l >> bit0) ^ (h * 0xD6E8FEB86659FD93ull);
        if (q == ~0ull) q--;
        uint32_t s = (uint32_t)((q * 0x9E3779B97F4A7C15ull) >> 50);  // 14 bits
        for (;;) {
            const unsigned long long old = atomicCAS(&slot[s], ~0ull, q);
            if (old == ~0ull) break;
            if (old == q) {
                found++;
                same = max(same, atomicAdd(&more[s], 1u) + 2u);
                break;
            }
            s = (s + 1) & (TW_SLOTS - 1);
        }
    }
    found = __reduce_add_sync(0xffffffffu, found);
    same = __reduce_max_sync(0xffffffffu, same);
    if ((threadIdx.x & 31) == 0 && found) {
        atomicAdd(&twins[blockIdx.y], (unsigned long long)found);
        atomicMax(&most[blockIdx.y], (unsigned long long)same);
    }
}

// Runs of equal prefixes of 2 to FX_RUN elements into the order of the whole
// key; the starts of longer ones go to the list.  A run belongs to the tile it
// starts in, which may move its elements beyond the tile's end while the next
// tile reads them: only their prefixes count there, and those are equal.  What
// bounds it is the read of the keys and, with many short runs, the moved ids (16M
// elements of the hetero rows' 8 tables: 0.26 ms; the passes it replaces took 1.1).
__global__ void __launch_bounds__(RS_THREADS) k_rs_settle(uint64_t *__restrict__ lo, uint64_t *__restrict__ hi,
                                                          uint32_t *__restrict__ v, int64_t m, int bit0,
                                                          int64_t *__restrict__ list,
                                                          unsigned long long *__restrict__ nlist) {
    extern __shared__ uint64_t fx_sm[];  // elements t0 - 1 .. t0 + RS_TILE + FX_RUN - 1
    constexpr int SPAN = RS_TILE + 1 + FX_RUN;
    uint64_t *sl = fx_sm, *sh = fx_sm + SPAN;
    const int64_t so = (int64_t)blockIdx.y * m, t0 = (int64_t)blockIdx.x * RS_TILE;
    const int64_t left = m - t0;  // elements from t0 on
    for (int e = threadIdx.x; e < SPAN; e += RS_THREADS) {
        const int64_t p = t0 - 1 + e;
        if (p >= 0 && p < m) {
            sl[e] = lo[so + p];
            sh[e] = hi[so + p];
        }
    }
    __syncthreads();
    const int cnt = (int)min((int64_t)RS_TILE, left), lim = (int)min((int64_t)(RS_TILE + FX_RUN), left);
    for (int e = threadIdx.x; e < cnt; e += RS_THREADS) {
        // element e of the tile at position e + 1
        const uint64_t l = sl[e + 1], h = sh[e + 1];
        if ((t0 + e > 0 && same_prefix(sl[e], sh[e], l, h, bit0)) || e + 1 >= lim ||
            !same_prefix(sl[e + 2], sh[e + 2], l, h, bit0))
            continue;
        int len = 2;
        while (len <= FX_RUN && e + len < lim && same_prefix(sl[e + 1 + len], sh[e + 1 + len], l, h, bit0))
            len++;
        if (len > FX_RUN) {
            list[atomicAdd(nlist, 1ull)] = so + t0 + e;
            continue;
        }
        // insertion; only this thread touches the run's keys and ids
        uint32_t *ids = v + so + t0 + e;
        bool moved = false;
        for (int i = 1; i < len; i++) {
            const uint64_t kl = sl[e + 1 + i], kh = sh[e + 1 + i];
            auto above = [&](int j) { return sh[e + 1 + j] != kh ? sh[e + 1 + j] > kh : sl[e + 1 + j] > kl; };
            if (!above(i - 1)) continue;
            const uint32_t id = ids[i];
            int j = i;
            for (; j > 0 && above(j - 1); j--) {
                sl[e + 1 + j] = sl[e + j];
                sh[e + 1 + j] = sh[e + j];
                ids[j] = ids[j - 1];
            }
            sl[e + 1 + j] = kl;
            sh[e + 1 + j] = kh;
            ids[j] = id;
            moved = true;
        }
        if (moved)
            for (int i = 0; i < len; i++) {
                lo[so + t0 + e + i] = sl[e + 1 + i];
                hi[so + t0 + e + i] = sh[e + 1 + i];
            }
    }
}

// The listed runs, a block each: least significant digit first over the bits
// below the prefix, between the sorted buffers and the spare ones.
constexpr int FL_ITEMS = 4;
__global__ void __launch_bounds__(RB_THREADS) k_rs_settle_long(uint64_t *lo, uint64_t *hi,
                                                               uint32_t *v, uint64_t *lo2,
                                                               uint64_t *hi2, uint32_t *v2,
                                                               int64_t m, int bit0, const int64_t *__restrict__ list,
                                                               const unsigned long long *__restrict__ nlist) {
    __shared__ uint32_t whist[RB_WARPS][256];
    __shared__ uint32_t at[256];
    __shared__ uint32_t wsum[32];
    const int t = threadIdx.x, warp = t >> 5, lane = t & 31;
    const uint32_t lt = (1u << lane) - 1;
    const int64_t nl = (int64_t)*nlist;
    for (int64_t r = blockIdx.x; r < nl; r += gridDim.x) {
        const int64_t p0 = list[r], room = (p0 / m + 1) * m - p0;
        const uint64_t l0 = lo[p0], h0 = hi[p0];
        int64_t len = 0;
        for (;;) {
            const int64_t p = len + t;
            const int c = __syncthreads_count(p < room &&
                                              same_prefix(lo[p0 + p], hi[p0 + p], l0, h0, bit0));
            len += c;
            if (c < RB_THREADS) break;
        }
        int pass = 0;
        for (int sh = 0; sh < bit0; sh += 8, pass++) {
            const uint64_t *sl = ((pass & 1) ? lo2 : lo) + p0, *shh = ((pass & 1) ? hi2 : hi) + p0;
            const uint32_t *sv = ((pass & 1) ? v2 : v) + p0;
            uint64_t *dl = ((pass & 1) ? lo : lo2) + p0, *dh = ((pass & 1) ? hi : hi2) + p0;
            uint32_t *dv = ((pass & 1) ? v : v2) + p0;
            auto digit = [&](uint64_t l, uint64_t h) { return (uint32_t)(((sh >= 64 ? h : l) >> (sh & 63)) & 0xFFu); };
            if (t < 256) at[t] = 0;
            __syncthreads();
            for (int64_t p = t; p < len; p += RB_THREADS) atomicAdd(&at[digit(sl[p], shh[p])], 1u);
            __syncthreads();
            uint32_t tot;
            const uint32_t ex = block_excl_scan<RB_THREADS>(t < 256 ? at[t] : 0u, &tot, wsum);
            if (t < 256) at[t] = ex;
            for (int64_t q0 = 0; q0 < len; q0 += RB_THREADS * FL_ITEMS) {
                for (int e = t; e < RB_WARPS * 256; e += RB_THREADS) whist[e >> 8][e & 255] = 0;
                __syncthreads();
                uint32_t dr[FL_ITEMS];
#pragma unroll
                for (int i = 0; i < FL_ITEMS; i++) {
                    const int64_t p = q0 + warp * (FL_ITEMS * 32) + i * 32 + lane;
                    const uint32_t d = p < len ? digit(sl[p], shh[p]) : 256u;
                    const uint32_t peers = __match_any_sync(0xffffffffu, d);
                    const int leader = __ffs(peers) - 1;
                    uint32_t old = 0;
                    if (lane == leader && d < 256) {
                        old = whist[warp][d];
                        whist[warp][d] = old + __popc(peers);
                    }
                    old = __shfl_sync(0xffffffffu, old, leader);
                    dr[i] = d | ((old + __popc(peers & lt)) << 9);
                }
                __syncthreads();
                if (t < 256) {
                    uint32_t run = at[t];
#pragma unroll
                    for (int w = 0; w < RB_WARPS; w++) {
                        const uint32_t c = whist[w][t];
                        whist[w][t] = run;
                        run += c;
                    }
                    at[t] = run;
                }
                __syncthreads();
#pragma unroll
                for (int i = 0; i < FL_ITEMS; i++) {
                    const int64_t p = q0 + warp * (FL_ITEMS * 32) + i * 32 + lane;
                    const uint32_t d = dr[i] & 511u;
                    if (d < 256) {
                        const uint32_t o = whist[warp][d] + (dr[i] >> 9);
                        dl[o] = sl[p];
                        dh[o] = shh[p];
                        dv[o] = sv[p];
                    }
                }
                __syncthreads();
            }
        }
        if (pass & 1)
            for (int64_t p = t; p < len; p += RB_THREADS) {
                lo[p0 + p] = lo2[p0 + p];
                hi[p0 + p] = hi2[p0 + p];
                v[p0 + p] = v2[p0 + p];
            }
        __syncthreads();
    }
}

// ---- run detection ---------------------------------------------------------
// a run starts where the key (lo, hi) or the optional tag changes
__device__ __forceinline__ bool run_start_at(const uint64_t *lo, const uint64_t *hi, const uint32_t *tag, int64_t p) {
    if (p == 0) return true;
    if (lo[p] != lo[p - 1]) return true;
    if (tag != nullptr && tag[p] != tag[p - 1]) return true;
    return hi != nullptr && hi[p] != hi[p - 1];
}

__global__ void __launch_bounds__(RS_THREADS) k_runs_count(const uint64_t *__restrict__ lo,
                                                           const uint64_t *__restrict__ hi,
                                                           const uint32_t *__restrict__ tag,
                                                           int64_t m, int tiles,
                                                           uint32_t *__restrict__ tile_cnt) {
    __shared__ uint32_t wsum[32];
    const int seg = blockIdx.y, tile = blockIdx.x;
    const uint64_t *l = lo + (int64_t)seg * m;
    const uint64_t *h = hi ? hi + (int64_t)seg * m : nullptr;
    const uint32_t *g = tag ? tag + (int64_t)seg * m : nullptr;
    const int64_t p0 = (int64_t)tile * RS_TILE + (int64_t)threadIdx.x * RS_ITEMS;
    uint32_t c = 0;
    for (int i = 0; i < RS_ITEMS; i++) {
        int64_t p = p0 + i;
        if (p < m && run_start_at(l, h, g, p)) c++;
    }
    uint32_t tot;
    block_excl_scan<RS_THREADS>(c, &tot, wsum);
    if (threadIdx.x == 0) tile_cnt[(int64_t)seg * tiles + tile] = tot;
}

__global__ void __launch_bounds__(RS_THREADS)
    k_runs_emit(const uint64_t *__restrict__ lo, const uint64_t *__restrict__ hi, const uint32_t *__restrict__ tag,
                int64_t m, int tiles, const uint32_t *__restrict__ tile_off, const int64_t *__restrict__ runs,
                int32_t *__restrict__ rank, int64_t *__restrict__ run_start) {
    __shared__ uint32_t wsum[32];
    const int seg = blockIdx.y, tile = blockIdx.x;
    const uint64_t *l = lo + (int64_t)seg * m;
    const uint64_t *h = hi ? hi + (int64_t)seg * m : nullptr;
    const uint32_t *g = tag ? tag + (int64_t)seg * m : nullptr;
    int64_t *rs = run_start + (int64_t)seg * (m + 1);
    const int64_t p0 = (int64_t)tile * RS_TILE + (int64_t)threadIdx.x * RS_ITEMS;
    uint32_t flags = 0, c = 0;
    for (int i = 0; i < RS_ITEMS; i++) {
        int64_t p = p0 + i;
        if (p < m && run_start_at(l, h, g, p)) {
            flags |= 1u << i;
            c++;
        }
    }
    uint32_t tot;
    uint32_t ex = block_excl_scan<RS_THREADS>(c, &tot, wsum) + tile_off[(int64_t)seg * tiles + tile];
    // rank of position p = (number of starts at positions <= p) - 1
    int64_t r = (int64_t)ex - 1;
    for (int i = 0; i < RS_ITEMS; i++) {
        int64_t p = p0 + i;
        if (p >= m) break;
        if (flags >> i & 1u) {
            r++;
            rs[r] = p;
        }
        if (rank) rank[(int64_t)seg * m + p] = (int32_t)r;
    }
    if (tile == 0 && threadIdx.x == 0) rs[runs[seg]] = m;
}

// Bucket formation from sorted segments in one pass: position p of segment
// seg (key-sorted, ids[] the object ids in that order) belongs to run r;
// the object's bucket id in its table is r, and a run start records the
// run's global offset.  Writes obj_bucket[seg][ids[p]] = r and, at starts,
// boff[base[seg] + r] = seg * m + p; boff[NB] = S * m closes the list.
// The tile's keys and ids are first copied to shared memory with coalesced
// loads (a thread then walks RS_ITEMS consecutive positions there); the key
// before the tile comes along for the first run-start test.
__global__ void __launch_bounds__(RS_THREADS)
    k_runs_buckets(const uint64_t *__restrict__ lo, const uint64_t *__restrict__ hi, int64_t m, int tiles,
                   const uint32_t *__restrict__ tile_off, const uint32_t *__restrict__ ids,
                   const int64_t *__restrict__ base, int32_t *__restrict__ obj_bucket,
                   int64_t *__restrict__ boff, int64_t NB) {
    extern __shared__ uint64_t rb_sm[];  // lo [RS_TILE + 1], hi [RS_TILE + 1] (when hi), ids [RS_TILE]
    __shared__ uint32_t wsum[32];
    const int seg = blockIdx.y, tile = blockIdx.x;
    const int64_t so = (int64_t)seg * m;
    const uint64_t *l = lo + so;
    const uint64_t *h = hi ? hi + so : nullptr;
    uint64_t *sl = rb_sm, *sh = rb_sm + (RS_TILE + 1);
    uint32_t *sid = reinterpret_cast<uint32_t *>(rb_sm + (h ? 2 : 1) * (RS_TILE + 1));
    const int64_t t0 = (int64_t)tile * RS_TILE;
    const int cnt = (int)min((int64_t)RS_TILE, m - t0);
    for (int e = threadIdx.x; e < cnt; e += RS_THREADS) {
        sl[e + 1] = l[t0 + e];
        if (h) sh[e + 1] = h[t0 + e];
        sid[e] = ids[so + t0 + e];
    }
    if (threadIdx.x == 0 && t0 > 0) {
        sl[0] = l[t0 - 1];
        if (h) sh[0] = h[t0 - 1];
    }
    __syncthreads();
    const int e0 = threadIdx.x * RS_ITEMS;
    uint32_t flags = 0, c = 0;
    for (int i = 0; i < RS_ITEMS; i++) {
        const int e = e0 + i;
        if (e < cnt && (t0 + e == 0 || sl[e + 1] != sl[e] || (h && sh[e + 1] != sh[e]))) {
            flags |= 1u << i;
            c++;
        }
    }
    uint32_t tot;
    const uint32_t ex = block_excl_scan<RS_THREADS>(c, &tot, wsum) + tile_off[(int64_t)seg * tiles + tile];
    int64_t r = (int64_t)ex - 1;
    const int64_t bb = base[seg];
    for (int i = 0; i < RS_ITEMS; i++) {
        const int e = e0 + i;
        if (e >= cnt) break;
        if (flags >> i & 1u) {
            r++;
            boff[bb + r] = so + t0 + e;
        }
        obj_bucket[so + sid[e]] = (int32_t)r;
    }
    if (seg == 0 && tile == 0 && threadIdx.x == 0) boff[NB] = (int64_t)gridDim.y * m;
}

// ---- generic int64 exclusive scan -----------------------------------------
__global__ void __launch_bounds__(RS_THREADS) k_i64_tile_sum(const int64_t *__restrict__ in,
                                                             int64_t n, int64_t *__restrict__ sums) {
    __shared__ int64_t red[RS_THREADS];
    // the tile's sum in any order (integers): lane-contiguous, coalesced loads
    const int64_t t0 = (int64_t)blockIdx.x * RS_TILE;
    int64_t s = 0;
    for (int i = 0; i < RS_ITEMS; i++) {
        const int64_t p = t0 + (int64_t)i * RS_THREADS + threadIdx.x;
        if (p < n) s += in[p];
    }
    red[threadIdx.x] = s;
    __syncthreads();
    for (int o = RS_THREADS / 2; o > 0; o >>= 1) {
        if (threadIdx.x < o) red[threadIdx.x] += red[threadIdx.x + o];
        __syncthreads();
    }
    if (threadIdx.x == 0) sums[blockIdx.x] = red[0];
}

// single block: exclusive scan of `n` int64 in place, total -> *total
__global__ void __launch_bounds__(1024) k_i64_scan_small(int64_t *__restrict__ a, int64_t n,
                                                         int64_t *__restrict__ total) {
    __shared__ int64_t buf[1024];
    int64_t carry = 0;
    for (int64_t base = 0; base < n; base += 1024) {
        int64_t p = base + threadIdx.x;
        int64_t v = p < n ? a[p] : 0;
        buf[threadIdx.x] = v;
        __syncthreads();
        for (int o = 1; o < 1024; o <<= 1) {
            int64_t y = threadIdx.x >= o ? buf[threadIdx.x - o] : 0;
            __syncthreads();
            buf[threadIdx.x] += y;
            __syncthreads();
        }
        if (p < n) a[p] = carry + buf[threadIdx.x] - v;
        carry += buf[1023];
        __syncthreads();
    }
    if (threadIdx.x == 0 && total) *total = carry;
}

__global__ void __launch_bounds__(RS_THREADS) k_i64_tile_apply(const int64_t *__restrict__ in,
                                                               int64_t *__restrict__ out, int64_t n,
                                                               const int64_t *__restrict__ sums) {
    __shared__ int64_t red[RS_THREADS];
    __shared__ int64_t tv[RS_TILE];  // the tile, loaded and stored coalesced
    const int64_t t0 = (int64_t)blockIdx.x * RS_TILE;
    const int cnt = (int)min((int64_t)RS_TILE, n - t0);
    for (int e = threadIdx.x; e < RS_TILE; e += RS_THREADS) tv[e] = e < cnt ? in[t0 + e] : 0;
    __syncthreads();
    const int e0 = threadIdx.x * RS_ITEMS;
    int64_t v[RS_ITEMS];
    int64_t s = 0;
    for (int i = 0; i < RS_ITEMS; i++) {
        v[i] = tv[e0 + i];
        s += v[i];
    }
    red[threadIdx.x] = s;
    __syncthreads();
    // Hillis-Steele inclusive scan over the 256 thread sums
    for (int o = 1; o < RS_THREADS; o <<= 1) {
        int64_t y = threadIdx.x >= o ? red[threadIdx.x - o] : 0;
        __syncthreads();
        red[threadIdx.x] += y;
        __syncthreads();
    }
    int64_t ex = red[threadIdx.x] - s + sums[blockIdx.x];
    for (int i = 0; i < RS_ITEMS; i++) {
        tv[e0 + i] = ex;
        ex += v[i];
    }
    __syncthreads();
    for (int e = threadIdx.x; e < cnt; e += RS_THREADS) out[t0 + e] = tv[e];
}

// the same for up to SCAN_ONE values, what a block holds in registers, by one
// block (one launch instead of three; with the fills of small sorts, the
// 20,000 x 32 pipeline 1.98 -> 1.85 ms): thread t the values 16 t .. 16 t + 15
constexpr int SCAN_ONE = 16384;
__global__ void __launch_bounds__(1024) k_i64_scan_one(const int64_t *__restrict__ in, int64_t *__restrict__ out, int n,
                                                       int64_t *__restrict__ total) {
    __shared__ int64_t s_warp[32];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    int64_t v[16], s = 0;
#pragma unroll
    for (int i = 0; i < 16; i++) {
        v[i] = 16 * t + i < n ? in[16 * t + i] : 0;
        s += v[i];
    }
    int64_t x = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int64_t y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
    }
    if (lane == 31) s_warp[w] = x;
    __syncthreads();
    if (w == 0) {
        int64_t z = s_warp[lane];
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int64_t y = __shfl_up_sync(0xffffffffu, z, o);
            if (lane >= o) z += y;
        }
        s_warp[lane] = z;
    }
    __syncthreads();
    int64_t ex = x - s + (w ? s_warp[w - 1] : 0);
#pragma unroll
    for (int i = 0; i < 16; i++) {
        if (16 * t + i < n) out[16 * t + i] = ex;
        ex += v[i];
    }
    if (t == 0 && total) *total = s_warp[31];
}

}  // namespace

geek_status set_error(geek_ctx *ctx, geek_status st, const char *fmt, ...) {
    if (ctx) {
        char buf[512];
        va_list ap;
        va_start(ap, fmt);
        vsnprintf(buf, sizeof buf, fmt, ap);
        va_end(ap);
        ctx->last_error = buf;
    }
    return st;
}

geek_status sort_err_word(geek_ctx *ctx) {
    if (ctx->sort_err) return GEEK_OK;
    GK_CUDA(ctx, cudaMalloc((void **)&ctx->sort_err, sizeof(int)));
    GK_CUDA(ctx, cudaMemset(ctx->sort_err, 0, sizeof(int)));
    return GEEK_OK;
}

geek_status sort_err_fetch(geek_ctx *ctx, int *h, cudaStream_t st) {
    *h = 0;
    if (!ctx->sort_err || ctx->capturing) return GEEK_OK;
    GK_CUDA(ctx, cudaMemcpyAsync(h, ctx->sort_err, sizeof *h, cudaMemcpyDeviceToHost, st));
    return GEEK_OK;
}

geek_status sort_err_eval(geek_ctx *ctx, const int *h, cudaStream_t st) {
    if (!*h) return GEEK_OK;
    GK_CUDA(ctx, cudaMemsetAsync(ctx->sort_err, 0, sizeof(int), st));
    return set_error(ctx, (geek_status)*h, "radix sort: a look-back wait timed out");
}

geek_status sort_err_check(geek_ctx *ctx, cudaStream_t st) {
    if (ctx->capturing) return GEEK_OK;
    int h = 0;
    GK_TRY(sort_err_fetch(ctx, &h, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    return sort_err_eval(ctx, &h, st);
}

geek_status radix_sort_segments(geek_ctx *ctx, Scratch &scr, int S, int64_t m, uint64_t **key_lo,
                                uint64_t **key_hi, uint32_t **vals, int nbits, cudaStream_t st, int bit0, bool iota, SortSpare *spare) {
    if (S <= 0 || m < 1) return GEEK_OK;
    if (m == 1 && iota) GK_CUDA(ctx, cudaMemsetAsync(*vals, 0, sizeof(uint32_t) * S, st));
    if (m == 1 || nbits <= bit0) return GEEK_OK;
    if (S > 65535) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "radix sort: %d segments", S);
    if (m > (int64_t)LB_MASK) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "radix sort: segment too long");
    if ((int64_t)S * ceil_div(m, RS_TILE) > 0xFFFFFFFFLL)
        return set_error(ctx, GEEK_ERR_UNSUPPORTED, "radix sort: too many tiles");
    const bool hi = nbits > 64;
    if (hi && !(key_hi && *key_hi)) return set_error(ctx, GEEK_ERR_INVALID, "radix sort: missing hi word");
    const bool hv = vals && *vals;
    const int npass = (nbits - bit0 + 7) / 8;
    if (m <= RB_MAX) {
        const size_t smem = (size_t)m * ((hi ? 16 : 8) + (hv ? 4 : 0));
        EvTimer tk(ctx, "kernel.rs_scatter", st);
        tk.work = 2.0 * (double)S * m * ((hi ? 16 : 8) + (hv ? 4 : 0)) * npass;
        GK_COUNT();
        auto run = [&](auto *k) -> geek_status {
            GK_CUDA(ctx, cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, RB_MAX * 20));
            k<<<S, RB_THREADS, smem, st>>>(*key_lo, hi ? *key_hi : nullptr, hv ? *vals : nullptr, (int)m, bit0, npass, iota);
            GK_LAUNCH(ctx);
            return GEEK_OK;
        };
        if (hi && hv) return run(k_rs_block<true, true>);
        if (hi) return run(k_rs_block<true, false>);
        if (hv) return run(k_rs_block<false, true>);
        return run(k_rs_block<false, false>);
    }
    const int tiles = (int)ceil_div(m, RS_TILE);
    const int64_t total = (int64_t)S * m;
    uint64_t *lo2 = nullptr, *hi2 = nullptr;
    uint32_t *v2 = nullptr;
    GK_TRY(scr.alloc(&lo2, total));
    if (hi) GK_TRY(scr.alloc(&hi2, total));
    if (hv) GK_TRY(scr.alloc(&v2, total));
    // iota: the first pass reads no values, so its output can be the buffer
    // that makes *vals the last pass's
    const bool odd = npass & 1;
    uint64_t *alo = *key_lo, *ahi = hi ? *key_hi : nullptr, *blo = lo2, *bhi = hi2;
    uint32_t *av = hv ? *vals : nullptr, *bv = v2;
    if (iota && odd) std::swap(av, bv);
    const size_t stage = (size_t)RS_TILE * ((hi ? 16 : 8) + (hv ? 4 : 0));
    static bool attr_done = false;
    if (!attr_done) {
        const int mx = RS_TILE * 20;
        GK_CUDA(ctx, cudaFuncSetAttribute(k_rs_onesweep<true, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
        GK_CUDA(ctx, cudaFuncSetAttribute(k_rs_onesweep<true, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
        GK_CUDA(ctx, cudaFuncSetAttribute(k_rs_onesweep<false, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
        GK_CUDA(ctx, cudaFuncSetAttribute(k_rs_onesweep<false, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, mx));
        GK_CUDA(ctx, cudaFuncSetAttribute(k_rs_hist_all, cudaFuncAttributeMaxDynamicSharedMemorySize, 4 * 16 * 256 * 4));
        attr_done = true;
    }
    // all digit offsets from one read of the keys
    // digit totals, then per pass the look-back words and the ticket: small
    // sorts clear all passes' words with the totals (one fill instead of npass
    // + 1), larger ones reuse one pass's words, cleared before each
    uint32_t *dbase_all, *look;
    const size_t nd = (size_t)S * npass * 256, nl = (size_t)S * tiles * 256 + 32;
    const bool one_fill = nl * npass <= ((size_t)4 << 20);  // 16 MB
    GK_TRY(scr.alloc(&dbase_all, nd + (one_fill ? npass : 1) * nl));
    look = dbase_all + nd;
    GK_TRY(sort_err_word(ctx));
    GK_CUDA(ctx, cudaMemsetAsync(dbase_all, 0, sizeof(uint32_t) * (nd + (one_fill ? npass * nl : 0)), st));
    {
        // few segments take more blocks each, so that the chip is full (the sorts
        // of the 256-instance batch, one segment: 5.6 -> 1.6 ms)
        const int hb = (int)std::min<int64_t>(std::max(HIST_BLOCKS_PER_SEG, 6 * ctx->num_sms / S), ceil_div(m, 256 * 16));
        GK_COUNT();
        k_rs_hist_all<<<dim3(std::max(hb, 1), S), 256, (size_t)4 * npass * 256 * 4, st>>>(alo, hi ? ahi : nullptr, m, bit0,
                                                                                        npass, dbase_all);
        GK_LAUNCH(ctx);
        GK_COUNT();
        k_rs_base_all<<<S * npass, 256, 0, st>>>(dbase_all);
        GK_LAUNCH(ctx);
    }
    const int64_t nblocks = (int64_t)S * tiles;
    for (int q = 0; q < npass; q++) {
        const int sh = bit0 + q * 8, dsel = sh >= 64, sv = sh & 63;
        if (!one_fill) GK_CUDA(ctx, cudaMemsetAsync(look, 0, sizeof(uint32_t) * nl, st));
        uint32_t *const lk = look + (one_fill ? q * nl : 0), *const ticket = lk + (nl - 32);
        EvTimer tk(ctx, "kernel.rs_scatter", st);
        tk.work = 2.0 * (double)total * ((hi ? 16 : 8) + (hv ? 4 : 0));
        GK_COUNT();
#define RS_OS(H, V)                                                                                              \
    k_rs_onesweep<H, V><<<(unsigned)nblocks, RS_THREADS, stage, st>>>(alo, ahi, iota && q == 0 ? nullptr : av, blo, bhi, bv, m, \
                                                                      tiles, dsel, sv, dbase_all + (size_t)q * 256, npass * 256, lk, \
                                                                      ticket, ctx->sort_err, ctx->lb_wait_ns, ctx->stall_tile)
        if (hi && hv) RS_OS(true, true);
        else if (hi) RS_OS(true, false);
        else if (hv) RS_OS(false, true);
        else RS_OS(false, false);
#undef RS_OS
        GK_LAUNCH(ctx);
        std::swap(alo, blo);
        std::swap(ahi, bhi);
        std::swap(av, bv);
    }
    if (odd && iota) {  // the values are in *vals, the keys change buffers
        *key_lo = alo;
        if (hi) *key_hi = ahi;
    } else if (odd) {  // result lives in the scratch buffers: copy back
        GK_CUDA(ctx, cudaMemcpyAsync(*key_lo, alo, total * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
        if (hi) GK_CUDA(ctx, cudaMemcpyAsync(*key_hi, ahi, total * sizeof(uint64_t), cudaMemcpyDeviceToDevice, st));
        if (hv) GK_CUDA(ctx, cudaMemcpyAsync(*vals, av, total * sizeof(uint32_t), cudaMemcpyDeviceToDevice, st));
    }
    if (spare) *spare = SortSpare{blo, bhi, bv};
    return GEEK_OK;
}

geek_status sort_ids(geek_ctx *ctx, Scratch &scr, int S, int64_t m, uint64_t **key_lo, uint64_t **key_hi,
                     uint32_t **ids, int nbits, cudaStream_t st) {
    // The upper bits alone for keys of two words, where that saves three passes or
    // more and the sample's cost (a launch and a wait, some 50 us) is small beside
    // them; log2 m + 2 bits are the fewest that can do.  For one-word keys it gives
    // nothing: 16 tables of 2M 60-bit keys saved two of eight passes (0.41 ms) and
    // paid 0.36 ms for sampling and settling.
    const int full = (nbits + 7) / 8, np0 = (bit_length_u64((uint64_t)m) + 2 + 7) / 8;
    const int widths = std::min(TW_WIDTHS, full - 3 - np0 + 1);
    if (nbits <= 64 || widths < 1 || S * m < (int64_t)8 << 20 || m < 4 * TW_SAMPLES)
        return radix_sort_segments(ctx, scr, S, m, key_lo, key_hi, ids, nbits, st, 0, true);
    int bit0 = (nbits - 8 * np0) & ~7;  // no digit across the words
    unsigned long long *cnt, h[2 * TW_WIDTHS];  // twins and most, then the listed runs
    GK_TRY(scr.alloc(&cnt, 2 * TW_WIDTHS + 1));
    GK_CUDA(ctx, cudaMemsetAsync(cnt, 0, (2 * TW_WIDTHS + 1) * sizeof *cnt, st));
    unsigned long long *const n_list = cnt + 2 * TW_WIDTHS;
    const size_t tw_smem = TW_SLOTS * (sizeof(unsigned long long) + sizeof(uint32_t));
    GK_CUDA(ctx, cudaFuncSetAttribute(k_rs_twins, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tw_smem));
    GK_COUNT();
    k_rs_twins<<<dim3(S, widths), 1024, tw_smem, st>>>(*key_lo, *key_hi, m, bit0, cnt, cnt + TW_WIDTHS);
    GK_LAUNCH(ctx);
    GK_CUDA(ctx, cudaMemcpyAsync(h, cnt, sizeof h, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    // An object with c others of its prefix has a twin among the samples with
    // probability c TW_SAMPLES / m.  With a quarter of another on average the
    // settling costs less than the passes it saves, even all in runs of 33 (a
    // block each); tables of large buckets take all the passes.  So do those with
    // one run of more than S m / 1,024 objects: a block settles an object in 18 ns,
    // the passes saved take 33 ps of it or more (64 tables of 131,072 objects, one
    // table a single run: 3.07 ms, 4.22 by settling; 8 tables of 2M with a run of
    // 2,000 each: 2.75 ms by settling, 4.75).
    auto settles = [&](int w) {
        return (double)h[w] * (double)m <= 0.25 * (double)S * TW_SAMPLES * TW_SAMPLES &&
               (double)h[TW_WIDTHS + w] * 1024 <= (double)S * TW_SAMPLES;
    };
    int w = 0;
    while (w < widths && !settles(w)) w++;
    if (w == widths) return radix_sort_segments(ctx, scr, S, m, key_lo, key_hi, ids, nbits, st, 0, true);
    bit0 -= 8 * w;
    SortSpare sp;
    GK_TRY(radix_sort_segments(ctx, scr, S, m, key_lo, key_hi, ids, nbits, st, bit0, true, &sp));
    int64_t *list;
    GK_TRY(scr.alloc(&list, (size_t)(S * m / (FX_RUN + 1) + 1)));
    const dim3 grid((unsigned)ceil_div(m, RS_TILE), S);
    const size_t smem = 2 * (size_t)(RS_TILE + 1 + FX_RUN) * sizeof(uint64_t);
    GK_COUNT();
    k_rs_settle<<<grid, RS_THREADS, smem, st>>>(*key_lo, *key_hi, *ids, m, bit0, list, n_list);
    GK_COUNT();
    k_rs_settle_long<<<2 * ctx->num_sms, RB_THREADS, 0, st>>>(*key_lo, *key_hi, *ids, sp.lo, sp.hi, sp.vals, m, bit0,
                                                              list, n_list);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

geek_status segment_runs(geek_ctx *ctx, Scratch &scr, int S, int64_t m, const uint64_t *key_lo,
                         const uint64_t *key_hi, int32_t *rank, int64_t *run_start, int64_t *runs,
                         cudaStream_t st) {
    return segment_runs_tagged(ctx, scr, S, m, key_lo, key_hi, nullptr, rank, run_start, runs, st);
}

geek_status segment_runs_tagged(geek_ctx *ctx, Scratch &scr, int S, int64_t m, const uint64_t *key_lo,
                                const uint64_t *key_hi, const uint32_t *tag, int32_t *rank, int64_t *run_start,
                                int64_t *runs, cudaStream_t st) {
    if (S <= 0) return GEEK_OK;
    if (m == 0) {
        GK_CUDA(ctx, cudaMemsetAsync(runs, 0, sizeof(int64_t) * S, st));
        GK_CUDA(ctx, cudaMemsetAsync(run_start, 0, sizeof(int64_t) * S, st));
        return GEEK_OK;
    }
    const int tiles = (int)ceil_div(m, RS_TILE);
    uint32_t *tile_cnt;
    GK_TRY(scr.alloc(&tile_cnt, (size_t)S * tiles));
    const dim3 grid(tiles, S);
    GK_COUNT();
    k_runs_count<<<grid, RS_THREADS, 0, st>>>(key_lo, key_hi, tag, m, tiles, tile_cnt);
    GK_COUNT();
    k_seg_scan_u32<<<S, 1024, 0, st>>>(tile_cnt, tiles, runs);
    GK_COUNT();
    k_runs_emit<<<grid, RS_THREADS, 0, st>>>(key_lo, key_hi, tag, m, tiles, tile_cnt, runs, rank, run_start);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

geek_status segment_buckets(geek_ctx *ctx, Scratch &scr, int S, int64_t m, const uint64_t *key_lo,
                            const uint64_t *key_hi, const uint32_t *ids, int32_t *obj_bucket, int64_t **boff_out,
                            std::vector<int64_t> &nb, int64_t *NB_out, cudaStream_t st) {
    nb.assign(S, 0);
    int64_t *runs;
    GK_TRY(scr.alloc(&runs, std::max(S, 1)));
    const int tiles = (int)std::max<int64_t>(1, ceil_div(m, RS_TILE));
    uint32_t *tile_cnt = nullptr;
    if (S > 0 && m > 0) {
        GK_TRY(scr.alloc(&tile_cnt, (size_t)S * tiles));
        GK_COUNT();
        k_runs_count<<<dim3(tiles, S), RS_THREADS, 0, st>>>(key_lo, key_hi, nullptr, m, tiles, tile_cnt);
        GK_COUNT();
        k_seg_scan_u32<<<S, 1024, 0, st>>>(tile_cnt, tiles, runs);
        GK_LAUNCH(ctx);
        GK_CUDA(ctx, cudaMemcpyAsync(nb.data(), runs, sizeof(int64_t) * S, cudaMemcpyDeviceToHost, st));
    }
    int sort_err = 0;
    GK_TRY(sort_err_fetch(ctx, &sort_err, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    GK_TRY(sort_err_eval(ctx, &sort_err, st));
    std::vector<int64_t> base(std::max(S, 1), 0);
    int64_t NB = 0;
    for (int l = 0; l < S; l++) {
        base[l] = NB;
        NB += nb[l];
    }
    int64_t *boff;
    cudaError_t e = cudaMallocAsync((void **)&boff, sizeof(int64_t) * (NB + 1), st);
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, GEEK_ERR_NOMEM, "bucket offsets: %s", cudaGetErrorString(e));
    }
    if (S == 0 || m == 0) {
        const int64_t sentinel = (int64_t)S * m;  // = 0
        GK_CUDA(ctx, cudaMemcpyAsync(boff + NB, &sentinel, sizeof sentinel, cudaMemcpyHostToDevice, st));
        GK_CUDA(ctx, cudaStreamSynchronize(st));
    } else {
        int64_t *d_base;
        GK_TRY(scr.alloc(&d_base, S));
        GK_CUDA(ctx, cudaMemcpyAsync(d_base, base.data(), sizeof(int64_t) * S, cudaMemcpyHostToDevice, st));
        GK_COUNT();
        const size_t rb_smem = (size_t)(key_hi ? 2 : 1) * (RS_TILE + 1) * sizeof(uint64_t) + RS_TILE * sizeof(uint32_t);
        static bool rb_attr = false;
        if (!rb_attr) {
            GK_CUDA(ctx, cudaFuncSetAttribute(k_runs_buckets, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                              (int)(2 * (RS_TILE + 1) * sizeof(uint64_t) + RS_TILE * sizeof(uint32_t))));
            rb_attr = true;
        }
        k_runs_buckets<<<dim3(tiles, S), RS_THREADS, rb_smem, st>>>(key_lo, key_hi, m, tiles, tile_cnt, ids, d_base,
                                                                   obj_bucket, boff, NB);
        GK_LAUNCH(ctx);
    }
    *boff_out = boff;
    *NB_out = NB;
    return GEEK_OK;
}

geek_status exclusive_scan_i64(geek_ctx *ctx, Scratch &scr, const int64_t *in, int64_t *out,
                               int64_t n, int64_t *total_dev, cudaStream_t st) {
    if (n <= 0) {
        if (total_dev) GK_CUDA(ctx, cudaMemsetAsync(total_dev, 0, sizeof(int64_t), st));
        return GEEK_OK;
    }
    if (n <= SCAN_ONE) {
        GK_COUNT();
        k_i64_scan_one<<<1, 1024, 0, st>>>(in, out, (int)n, total_dev);
        GK_LAUNCH(ctx);
        return GEEK_OK;
    }
    const int64_t tiles = ceil_div(n, RS_TILE);
    int64_t *sums;
    GK_TRY(scr.alloc(&sums, tiles));
    GK_COUNT();
    k_i64_tile_sum<<<(unsigned)tiles, RS_THREADS, 0, st>>>(in, n, sums);
    GK_COUNT();
    k_i64_scan_small<<<1, 1024, 0, st>>>(sums, tiles, total_dev);
    GK_COUNT();
    k_i64_tile_apply<<<(unsigned)tiles, RS_THREADS, 0, st>>>(in, out, n, sums);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}
