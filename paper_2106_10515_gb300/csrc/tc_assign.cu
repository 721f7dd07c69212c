// Dense one-pass assignment on the 5th-generation tensor cores (tcgen05).
//
// S = X C^T in BF16 with FP32 accumulation in tensor memory, fused with a
// running arg-min epilogue over centre tiles; the FP64 decision of the
// exact argmin (Eq. 1) is left to objects whose best and second-best
// approximate values are closer than the rigorous error window.
//
// Persistent kernel, one CTA per SM, 10 warps:
//   warp 0     TMA producer: X row tiles (a ring of 2 or 4 stages) and centre
//              tiles (2 to 8 stages, whole tiles or 64-column parts), 128-byte
//              swizzled, K-major, plus |c|^2 of each centre tile
//   warp 1     MMA issuer: tcgen05.mma.cta_group::1.kind::f16, M=128, N=256,
//              into one of two TMEM accumulators (2 x 256 columns)
//   warps 2-9  epilogue: tcgen05.ld of the accumulator, d' = |c|^2 - 2 s,
//              per-row best / second-best over the centres; each warp reads
//              its TMEM lane quarter (warp % 4) and one half of the columns
//              (each column group is an independent running minimum per
//              row, so fewer groups mean fewer new-best rescans)
// Every mbarrier wait is bounded: on expiry the kernel records
// GEEK_ERR_TIMEOUT, stops issuing work, drains its own copies and MMAs, frees
// its tensor memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cfloat>

#include "internal.cuh"
#include "tc_ptx.cuh"

// One instance of the (batched) assignment.  Device copies are read by the
// kernel; CUtensorMap's 64-byte alignment keeps every array element aligned.
struct TcInst {
    CUtensorMap tmA;             // Xb: {Kp, n} bf16, box {64, 128}
    CUtensorMap tmB;             // Cb = -2 c: {Kp, kpad} bf16, box {64, N}
    CUtensorMap tmX;             // |c|^2 columns: {16, kpad} bf16, box {16, N}, 32-byte swizzle
    const float *xnorm;          // n: upper bound of |x|
    const unsigned *cmax_bits;   // max over real centres of |c|^2 (FP32 bits)
    int32_t *labels;             // n
    int64_t n, k;
    int64_t row_base;            // global row of local row 0 (flag list entries)
    int ntiles_c, Kp, d, N;      // centre tiles of N columns, padded d, d, tile N
    int split;                   // stored as [hi | lo] pairs
};

// Per-instance conversion arguments (device copies).
struct TcXPrep {
    const float *x;
    int64_t ldx;
    int d, Kp;
    int split;          // 1: rows hold [bf16(x) | bf16(x - bf16(x))]
    __nv_bfloat16 *xb;  // n x Kp (x 2 when split)
};
struct TcCPrep {
    const double *c;    // k x d
    int64_t k, kpad;
    int d, Kp;
    int split;
    __nv_bfloat16 *cb;  // kpad x Kp (x 2 when split): -2 c
    __nv_bfloat16 *cbx; // kpad x 16: |c|^2 as bf16 hi, mid, lo, then zeros
    float *cn;          // kpad: |c|^2 in FP32 (for max |c|)
    unsigned *cmax_bits;
};

namespace {

constexpr int TC_M = 128;
constexpr int TC_N = 256;
constexpr int TC_KB = 64;  // bf16 elements per 128-byte swizzle row
constexpr int TC_EPI_WARPS = 8;                   // 2 per TMEM lane quarter
constexpr int TC_EPI_GROUPS = TC_EPI_WARPS / 4;     // column groups per tile
constexpr int TC_MISC = 2048;                       // barriers, TMEM slot, merge buffer
constexpr int TC_THREADS = 32 * (2 + TC_EPI_WARPS);
constexpr int TC_KP_MAX = 128;                      // d <= 128
constexpr int TC_A_STAGE = TC_M * TC_KP_MAX * 2;    // bytes of one X tile stage
constexpr int TC_B_STAGE = TC_N * TC_KP_MAX * 2;    // bytes of one centre tile stage
// split-BF16 mode: an X stage holds one k-block's [hi | lo] pair.  Two stages are
// the two k-blocks of a row tile of 128 columns, or two row tiles of 64; the
// centre ring's stages hold a whole [hi | lo] tile or, where that exceeds half
// the ring (N = 256, Kp = 128), one 64-column block of it, so that 256-wide
// tiles fit: 64-wide tiles, the widest whole ones at Kp = 128, read the X block
// from shared memory once per 64 columns (300,007 x 100, k = 1,999: 646 us,
// 256-wide 381 us).  Instances of a batch have few centre tiles per row tile, so
// the next row tile's X must be on its way early: with tiles of N Kp <= 8192
// the X ring takes four stages and the centre ring what is left, 64 KB (the
// 256-instance batch: 11.9 ms, with two X stages 16.7 ms).
constexpr uint32_t TC_TMEM_COLS = 512;

// EMIT: a wave of gathered flagged rows instead of an instance's own.  Slot s of
// the wave is row s of the gathered buffer; unit u (128 slots) belongs to
// instance unit_inst[u0 + u].
struct TcEmit {
    const CUtensorMap *tmG;      // gathered rows, box {64, 128}
    const float *lim;            // per slot: a centre up to this value is a candidate
    uint32_t *masks;             // per slot kw words: bit j = centre j is a candidate
    int kw;
    const int *unit_inst;
    const int *n_units;          // of all waves
    int64_t u0;                  // first unit of this wave
};
struct TcArgs {
    const TcInst *inst;
    const int2 *units;           // (instance, row tile); null: instance 0, unit = row tile
    int64_t nunits;
    int32_t *flag_rows;          // global rows whose argmin needs the exact decision
    float *flag_m;               // their smallest values (NaN: none finite), beside flag_rows
    unsigned long long *n_flag;
    int *err;
    int lg_ns;                   // log2 of the centre-tile ring's stages (1..3)
    int lg_nx;                   // log2 of the |c|^2 ring's stages: lg_ns, or 1 with tiles in parts
    int lg_na;                   // log2 of the X ring's stages (1 or, split, 2), 32 KB each
    TcEmit e;
};

// three-input minimum
__device__ __forceinline__ float min3f(float a, float b, float c) {
    float d;
    asm("min.f32 %0, %1, %2, %3;" : "=f"(d) : "f"(a), "f"(b), "f"(c));
    return d;
}

// Rigorous half-window of the BF16 path for one object.  The accumulator
// holds |c|^2 - 2 x_h.c_h summed by the tensor core: -2 c is exact in BF16,
// and |c|^2 enters as hi + mid + lo BF16 terms (within 2^-24 |c|^2) times one.
//   inputs rounded to bf16 (u_b = 2^-8):     2 (2 u_b + u_b^2) |x| cmax
//   |c|^2 split:                             2^-24 cmax^2
//   the tensor core's accumulation of the d + 3 products, bounded loosely
//   by (d + 19) 2^-21 of the sum of their magnitudes:
//                                            (d + 19) 2^-21 (2 |x| cmax + cmax^2)(1 + 2 u_b)
//   the FP64 reference's own error:          (d + 3) 2^-53 (|x| + cmax)^2
// times 1.01 for second-order terms.
__device__ __forceinline__ float window_bf16(float xn, float cmax, int d) {
    const float ub = 0.00390625f;
    const float xc = xn * cmax, c2 = cmax * cmax;
    const float e = 2.f * (2.f * ub + ub * ub) * xc + 5.9604645e-8f * c2 +
                    (float)(d + 19) * 4.76837158e-7f * (2.f * xc + c2) * (1.f + 2.f * ub);
    const float s = xn + cmax;
    const float e64 = (float)(d + 3) * 1.1102230e-16f * s * s;
    return 1.01f * (e + e64) + 1e-30f;
}

// Rigorous half-window of the split-BF16 path.  With x_h = bf16(x), x_l =
// bf16(x - x_h) (and the same for c), x.c - (x_h.c_h + x_l.c_h + x_h.c_l) =
// -(x - x_h - x_l).c_h - x_h.(c - c_h - c_l) + (x - x_h).(c - c_h), each
// term bounded by u_b^2 (1 + u_b) |x| |c|: input term 2 * 3 u_b^2 (1 + u_b)
// |x| cmax; the |c|^2 split 2^-24 cmax^2; the accumulation of 3d + 3
// products (3d + 19) 2^-21 (2 |x| cmax (1 + 4 u_b) + cmax^2 (1 + 2 u_b)); the
// FP64 reference term as in window_bf16; times 1.01.
__device__ __forceinline__ float window_bf16x3(float xn, float cmax, int d) {
    const float ub = 0.00390625f;
    const float xc = xn * cmax, c2 = cmax * cmax;
    const float e = 6.f * ub * ub * (1.f + ub) * xc + 5.9604645e-8f * c2 +
                    (float)(3 * d + 19) * 4.76837158e-7f * (2.f * xc * (1.f + 4.f * ub) + c2 * (1.f + 2.f * ub));
    const float s = xn + cmax;
    const float e64 = (float)(d + 3) * 1.1102230e-16f * s * s;
    return 1.01f * (e + e64) + 1e-30f;
}

// Running minimum of one warp's rows over NCH 32-column chunks of one
// accumulator tile (columns jb .. jb + 32 NCH - 1); the TMEM load of chunk
// ch + 1 is in flight while chunk ch is reduced.  Per row:
//   b1     the smallest value so far, found in the chunk saved in sv / sj
//   b2o    the smallest value outside that chunk
// A chunk with a new minimum is copied to sv (its index and second-smallest
// value are resolved once per row tile, see epi_resolve); any other chunk
// only lowers b2o.  So min(b2o, second smallest of sv) is exactly the
// runner-up over all columns.
template <int NCH>
__device__ __forceinline__ void epi_tile(uint32_t tbase, int64_t jb, float &b1, float &b2o, float (&sv)[32],
                                         int64_t &sj) {
    uint32_t ra[32], rb[32];
    tmem_ld32_async(tbase, ra);
    tmem_wait_ld();
#pragma unroll
    for (int ch = 0; ch < NCH; ch++) {
        if (ch + 1 < NCH) {
            if (ch & 1) tmem_ld32_async(tbase + (ch + 1) * 32, ra);
            else tmem_ld32_async(tbase + (ch + 1) * 32, rb);
        }
        const uint32_t *r = (ch & 1) ? rb : ra;
        float v[32];  // d' = |c|^2 - 2 x.c, straight from the accumulator
#pragma unroll
        for (int i = 0; i < 32; i++) v[i] = __uint_as_float(r[i]);
        float t11[11];
#pragma unroll
        for (int i = 0; i < 10; i++) t11[i] = min3f(v[3 * i], v[3 * i + 1], v[3 * i + 2]);
        t11[10] = fminf(v[30], v[31]);
        const float tm = fminf(min3f(min3f(t11[0], t11[1], t11[2]), min3f(t11[3], t11[4], t11[5]),
                                     min3f(t11[6], t11[7], t11[8])),
                               fminf(t11[9], t11[10]));
        if (tm < b1) {
            b2o = fminf(b2o, b1);  // the old best chunk is now "outside"
            b1 = tm;
#pragma unroll
            for (int i = 0; i < 32; i++) sv[i] = v[i];
            sj = jb + ch * 32;
        } else {
            b2o = fminf(b2o, tm);
        }
        if (ch + 1 < NCH) tmem_wait_ld();
    }
}

// The candidates of one warp's rows among NCH 32-column chunks: bit i of
// out[ch] = column jb + 32 ch + i is at most lim.
template <int NCH>
__device__ __forceinline__ void emit_tile(uint32_t tbase, float lim, uint32_t *__restrict__ out) {
    uint32_t ra[32], rb[32];
    tmem_ld32_async(tbase, ra);
    tmem_wait_ld();
#pragma unroll
    for (int ch = 0; ch < NCH; ch++) {
        if (ch + 1 < NCH) {
            if (ch & 1) tmem_ld32_async(tbase + (ch + 1) * 32, ra);
            else tmem_ld32_async(tbase + (ch + 1) * 32, rb);
        }
        const uint32_t *r = (ch & 1) ? rb : ra;
        float tm = FLT_MAX;
#pragma unroll
        for (int i = 0; i < 30; i += 3)
            tm = fminf(tm, min3f(__uint_as_float(r[i]), __uint_as_float(r[i + 1]), __uint_as_float(r[i + 2])));
        tm = min3f(tm, __uint_as_float(r[30]), __uint_as_float(r[31]));
        uint32_t m = 0;
        if (tm <= lim) {
#pragma unroll
            for (int i = 0; i < 32; i++) m |= (__uint_as_float(r[i]) <= lim ? 1u : 0u) << i;
        }
        out[ch] = m;
        if (ch + 1 < NCH) tmem_wait_ld();
    }
}

// Index (first position) of the minimum in the saved chunk and the exact
// runner-up over all columns.
__device__ __forceinline__ void epi_resolve(float b1, float b2o, const float (&sv)[32], int64_t sj, float &b2,
                                            int &i1) {
    if (sj < 0) {  // no finite value at all
        b2 = b2o;
        i1 = 0x7FFFFFFF;
        return;
    }
    int idx = 31;
#pragma unroll
    for (int i = 31; i >= 0; i--)
        if (sv[i] == b1) idx = i;
    float m2 = FLT_MAX;
#pragma unroll
    for (int i = 0; i < 32; i++) m2 = fminf(m2, i == idx ? FLT_MAX : sv[i]);
    b2 = fminf(b2o, m2);
    i1 = (int)(sj + idx);
}

// SPLIT = false: S = x_h . c_h, one BF16 product per element (window_bf16).
// SPLIT = true: x = x_h + x_l and c = c_h + c_l in BF16 pairs, S = x_h . c_h +
// x_l . c_h + x_h . c_l: three MMAs per k-step into the same accumulator
// (window_bf16x3, ~100x narrower).
// EMIT: the rows are gathered flagged rows and the epilogue writes, instead of
// the argmin, the mask of every row's candidates (units of the other mode's
// instances are left to the launch of that mode).
template <bool SPLIT, bool EMIT>
__global__ void __launch_bounds__(TC_THREADS, 1) k_assign_tc(const __grid_constant__ TcArgs A) {
    constexpr int A_ST = TC_A_STAGE;
    constexpr int KW = SPLIT ? 2 : 1;  // stored column blocks per k-block
    if (EMIT && (int64_t)*A.e.n_units <= A.e.u0) return;  // a wave past the flagged rows
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    const int NA = 1 << A.lg_na;
    uint8_t *sA0 = base, *sB0 = base + NA * TC_A_STAGE;
    uint64_t *bars = (uint64_t *)(base + 2 * TC_A_STAGE + 2 * TC_B_STAGE);
    uint64_t *full_a = bars, *empty_a = bars + 4, *full_acc = bars + 8, *empty_acc = bars + 10;  // X ring: up to 4
    uint64_t *done_bar = bars + 12, *full_b = bars + 13, *empty_b = bars + 21;  // centre ring: up to 8
    uint32_t *tmem_slot = (uint32_t *)(bars + 29);
    // the centre-tile ring: the same bytes cut into NS stages (narrower tiles,
    // more stages in flight)
    const int NS = 1 << A.lg_ns;
    const int BSTR = (2 * TC_B_STAGE - (NA - 2) * TC_A_STAGE) / NS, XSTR = (2 * TC_N * 32) >> A.lg_nx;
    // stored 64-column blocks per stage: the whole tile, or one (a part)
    auto blocks_of = [&](const TcInst &I) {
        const int all = KW * I.Kp / TC_KB;
        return SPLIT && all * I.N * 128 > BSTR ? 1 : all;
    };
    float *mrg = (float *)(bars + 32);  // [groups-1][128][3] results of column groups 1..
    // |c|^2 columns: an all-ones X block (128 x 16) and per stage the centres'
    // (hi, mid, lo, 0...) rows (N x 16), 32-byte swizzled; one extra K = 16
    // step adds |c|^2 to every accumulator column
    uint8_t *sOnes = base + 2 * TC_A_STAGE + 2 * TC_B_STAGE + TC_MISC;  // 4 KB
    uint8_t *sX0 = sOnes + TC_M * 32;                                   // [2][TC_N * 32]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 4; i++) {
            mbar_init(&full_a[i], 1);
            mbar_init(&empty_a[i], 1);
        }
        for (int i = 0; i < 2; i++) {
            mbar_init(&full_acc[i], 1);
            mbar_init(&empty_acc[i], TC_EPI_WARPS);
        }
        for (int i = 0; i < 8; i++) {
            mbar_init(&full_b[i], 1);
            mbar_init(&empty_b[i], 1);
        }
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    // the all-ones block (1.0 in BF16 everywhere, so its swizzle is moot)
    for (int e = threadIdx.x; e < TC_M * 32 / 4; e += blockDim.x)
        reinterpret_cast<uint32_t *>(sOnes)[e] = 0x3F803F80u;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(TC_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const int64_t nunits = EMIT ? max((int64_t)0, min(A.nunits, (int64_t)*A.e.n_units - A.e.u0)) : A.nunits;
    auto unit = [&](int64_t u) {
        if (EMIT) return make_int2(A.e.unit_inst[A.e.u0 + u], (int)u);
        return A.units ? A.units[u] : make_int2(0, (int)u);
    };

    // Every role walks the same unit sequence (unit u = blockIdx.x + j *
    // gridDim.x); an instance's Kp, N and centre-tile count fix the per-unit
    // copy sizes, MMA shape and epilogue width.
    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            uint64_t ct = 0, pt = 0, ac = 0;  // centre tiles, ring stages and X stages so far
            uint32_t issued_b[8] = {0, 0, 0, 0, 0, 0, 0, 0}, issued_a[4] = {0, 0, 0, 0};
            bool ok = true;
            for (int64_t u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
                const int2 un = unit(u);
                const TcInst &I = A.inst[un.x];
                if (EMIT && (I.split != 0) != SPLIT) continue;
                const int nkb = I.Kp / TC_KB, N = I.N;  // logical k-blocks
                const int all = KW * nkb, bps = blocks_of(I);
                // X: one stage with every k-block, or (split) a stage per
                // k-block with its hi and lo columns
                for (int c = 0; c < (SPLIT ? nkb : 1); c++, ac++) {
                    const int ab = (int)(ac & (uint64_t)(NA - 1));
                    const uint32_t ua = (uint32_t)(ac >> A.lg_na);
                    if (!(ok = mbar_wait(&empty_a[ab], (ua & 1) ^ 1, A.err))) break;
                    const int nb = SPLIT ? 2 : nkb;
                    mbar_expect_tx(&full_a[ab], (uint32_t)(nb * TC_M * 128));
                    for (int b = 0; b < nb; b++)
                        tma_load_2d(su32(sA0 + ab * A_ST + b * TC_M * 128), EMIT ? A.e.tmG : &I.tmA,
                                    SPLIT ? c * TC_KB + b * I.Kp : b * TC_KB, un.y * TC_M, &full_a[ab]);
                    issued_a[ab] = ua + 1;
                }
                for (int c = 0; c < I.ntiles_c && ok; c++, ct++)
                    for (int b0 = 0; b0 < all; b0 += bps, pt++) {
                        const int s = (int)(pt & (uint64_t)(NS - 1));
                        const uint32_t uu = (uint32_t)(pt >> A.lg_ns);
                        if (!(ok = mbar_wait(&empty_b[s], (uu & 1) ^ 1, A.err))) break;
                        mbar_expect_tx(&full_b[s], (uint32_t)(bps * N * 128) + (b0 == 0 ? (uint32_t)N * 32 : 0u));
                        // split: blocks in the order hi 0, lo 0, hi 1, lo 1
                        for (int b = 0; b < bps; b++) {
                            const int q = b0 + b;
                            tma_load_2d(su32(sB0 + s * BSTR + b * N * 128), &I.tmB,
                                        SPLIT ? (q >> 1) * TC_KB + (q & 1) * I.Kp : q * TC_KB, c * N, &full_b[s]);
                        }
                        if (b0 == 0)
                            tma_load_2d(su32(sX0 + (int)(ct & ((1u << A.lg_nx) - 1)) * XSTR), &I.tmX, 0, c * N, &full_b[s]);
                        issued_b[s] = uu + 1;
                    }
            }
            // drain: every copy this thread issued has landed
            for (int s = 0; s < NA; s++)
                if (issued_a[s]) mbar_wait(&full_a[s], (issued_a[s] - 1) & 1, A.err, true);
            for (int s = 0; s < NS; s++)
                if (issued_b[s]) mbar_wait(&full_b[s], (issued_b[s] - 1) & 1, A.err, true);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            uint64_t ct = 0, pt = 0, ac = 0;
            bool ok = true;
            for (int64_t u = blockIdx.x; u < nunits && ok; u += gridDim.x) {
                const int2 un = unit(u);
                const TcInst &I = A.inst[un.x];
                if (EMIT && (I.split != 0) != SPLIT) continue;
                const int nkb = I.Kp / TC_KB, N = I.N, d = I.d;  // logical k-blocks
                const int all = KW * nkb, bps = blocks_of(I);
                const uint32_t idesc = idesc_bf16(TC_M, N);
                for (int c = 0; c < I.ntiles_c && ok; c++, ct++) {
                    const int s = (int)(ct & 1);  // accumulator buffer
                    const uint32_t uu = (uint32_t)(ct >> 1);
                    const uint32_t dtm = tmem + (uint32_t)(s * TC_N);
                    if (bps == all) {
                        // the whole tile in one stage: few instructions per
                        // MMA (a 64-wide one takes 32 cycles)
                        const int sb = (int)(pt & (uint64_t)(NS - 1));
                        if (!(ok = mbar_wait(&full_b[sb], (uint32_t)(pt >> A.lg_ns) & 1, A.err))) break;
                        if (!(ok = mbar_wait(&empty_acc[s], (uu & 1) ^ 1, A.err))) break;
                        if (c == 0)
                            for (int q = 0; q < (SPLIT ? nkb : 1) && ok; q++)
                                ok = mbar_wait(&full_a[(ac + q) & (uint64_t)(NA - 1)], (uint32_t)((ac + q) >> A.lg_na) & 1,
                                               A.err);
                        if (!ok) break;
                        fence_after();
                        uint64_t db = sdesc(su32(sB0 + sb * BSTR));
                        const uint32_t bl = (uint32_t)(N * 128) >> 4;  // the next block, in descriptor units
                        for (int kb = 0; kb < nkb; kb++, db += KW * bl) {
                            const uint64_t at = SPLIT ? ac + kb : ac;
                            const uint64_t da =
                                sdesc(su32(sA0 + (int)(at & (uint64_t)(NA - 1)) * A_ST) + (SPLIT ? 0 : kb * TC_M * 128));
#pragma unroll
                            for (int ks = 0; ks < TC_KB / 16; ks++) {
                                if (kb * TC_KB + ks * 16 >= d) break;  // zeros from here on
                                mma_bf16(dtm, da + 2 * ks, db + 2 * ks, idesc, (kb | ks) != 0);
                                if (SPLIT) {  // x_l . c_h and x_h . c_l
                                    mma_bf16(dtm, da + (TC_M * 128 >> 4) + 2 * ks, db + 2 * ks, idesc, 1);
                                    mma_bf16(dtm, da + 2 * ks, db + bl + 2 * ks, idesc, 1);
                                }
                            }
                        }
                        // + |c|^2: ones (128 x 16) times the centres' (hi, mid, lo, 0...)
                        mma_bf16(dtm, sdesc32(su32(sOnes)),
                                 sdesc32(su32(sX0 + (int)(ct & ((1u << A.lg_nx) - 1)) * XSTR)), idesc, 1);
                        mma_commit(&empty_b[sb]);
                        if (SPLIT && c + 1 == I.ntiles_c)
                            for (int q = 0; q < nkb; q++) mma_commit(&empty_a[(ac + q) & (uint64_t)(NA - 1)]);
                        pt++;
                    } else {
                        // split, the tile in parts: hi 0, lo 0, hi 1, lo 1
                        for (int q = 0; q < all; q++, pt++) {
                            const int sb = (int)(pt & (uint64_t)(NS - 1)), kb = q >> 1;
                            const int ab = (int)((ac + kb) & (uint64_t)(NA - 1));  // X stage
                            if (!(ok = mbar_wait(&full_b[sb], (uint32_t)(pt >> A.lg_ns) & 1, A.err))) break;
                            if (q == 0 && !(ok = mbar_wait(&empty_acc[s], (uu & 1) ^ 1, A.err))) break;
                            if (c == 0 && (q & 1) == 0 &&
                                !(ok = mbar_wait(&full_a[ab], (uint32_t)((ac + kb) >> A.lg_na) & 1, A.err)))
                                break;
                            fence_after();
                            const uint64_t da = sdesc(su32(sA0 + ab * A_ST)), db = sdesc(su32(sB0 + sb * BSTR));
#pragma unroll
                            for (int ks = 0; ks < TC_KB / 16; ks++) {
                                if (kb * TC_KB + ks * 16 >= d) break;
                                mma_bf16(dtm, da + 2 * ks, db + 2 * ks, idesc, (q | ks) != 0);
                                // a hi block meets x_l too: x_h.c_h + x_l.c_h, then x_h.c_l
                                if ((q & 1) == 0) mma_bf16(dtm, da + (TC_M * 128 >> 4) + 2 * ks, db + 2 * ks, idesc, 1);
                            }
                            if (q == 0)
                                mma_bf16(dtm, sdesc32(su32(sOnes)),
                                         sdesc32(su32(sX0 + (int)(ct & ((1u << A.lg_nx) - 1)) * XSTR)), idesc, 1);
                            // X stage: last read of its k-block in the last centre tile
                            if ((q & 1) && c + 1 == I.ntiles_c) mma_commit(&empty_a[ab]);
                            mma_commit(&empty_b[sb]);
                        }
                    }
                    if (!ok) break;
                    mma_commit(&full_acc[s]);
                }
                if (!ok) break;
                if (!SPLIT) mma_commit(&empty_a[ac & (uint64_t)(NA - 1)]);
                ac += SPLIT ? nkb : 1;
            }
            // drain: all MMAs this thread issued have completed
            mma_commit(done_bar);
            mbar_wait(done_bar, 0, A.err, true);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue
        const int ew = warp - 2;
        const int q = warp & 3;     // TMEM lane quarter this warp may access
        const int h = ew >> 2;      // column group
        const int rloc = 32 * q + lane;
        uint64_t ct = 0;
        bool ok = true;
        for (int64_t u = blockIdx.x; u < nunits; u += gridDim.x) {
            const int2 un = unit(u);
            const TcInst &I = A.inst[un.x];
            if (EMIT && (I.split != 0) != SPLIT) continue;
            const int N = I.N;
            const int gcols = N / TC_EPI_GROUPS;  // columns of this warp's group
            const int nch = gcols / 32;           // 32-column chunks (1, 2 or 4)
            const int64_t row = (int64_t)un.y * TC_M + rloc;
            if (EMIT) {
                const float lim = A.e.lim[row];
                uint32_t *out = A.e.masks + row * A.e.kw;
                for (int c = 0; c < I.ntiles_c; c++, ct++) {
                    const int s = (int)(ct & 1);
                    const uint32_t uu = (uint32_t)(ct >> 1);
                    int w_ok = 0;
                    if (lane == 0 && ok) w_ok = mbar_wait(&full_acc[s], uu & 1, A.err);
                    w_ok = __shfl_sync(0xffffffffu, w_ok, 0);
                    ok = ok && w_ok;
                    if (ok) {
                        fence_after();
                        const uint32_t tbase = tmem + (uint32_t)(s * TC_N + h * gcols) + ((uint32_t)(32 * q) << 16);
                        uint32_t *o = out + (c * N + h * gcols) / 32;
                        if (nch == 4) emit_tile<4>(tbase, lim, o);
                        else if (nch == 2) emit_tile<2>(tbase, lim, o);
                        else emit_tile<1>(tbase, lim, o);
                        fence_before();
                    }
                    __syncwarp();
                    if (lane == 0) mbar_arrive(&empty_acc[s]);
                }
                continue;
            }
            const float xn = row < I.n ? I.xnorm[row] : 0.f;
            const float cmax = sqrtf(__uint_as_float(*I.cmax_bits)) * (1.f + 1e-5f);
            const float W = 2.f * (SPLIT ? window_bf16x3(xn, cmax, I.d) : window_bf16(xn, cmax, I.d));
            const float Wc = W * (1.f + 1e-6f);
            float b1 = FLT_MAX, b2o = FLT_MAX, sv[32];
            int64_t sj = -1;
            for (int c = 0; c < I.ntiles_c; c++, ct++) {
                const int s = (int)(ct & 1);
                const uint32_t uu = (uint32_t)(ct >> 1);
                int w_ok = 0;
                if (lane == 0 && ok) w_ok = mbar_wait(&full_acc[s], uu & 1, A.err);
                w_ok = __shfl_sync(0xffffffffu, w_ok, 0);
                ok = ok && w_ok;
                if (ok) {
                    fence_after();
                    const uint32_t tbase = tmem + (uint32_t)(s * TC_N + h * gcols) + ((uint32_t)(32 * q) << 16);
                    const int64_t jb = (int64_t)c * N + h * gcols;
                    if (nch == 4) epi_tile<4>(tbase, jb, b1, b2o, sv, sj);
                    else if (nch == 2) epi_tile<2>(tbase, jb, b1, b2o, sv, sj);
                    else epi_tile<1>(tbase, jb, b1, b2o, sv, sj);
                    fence_before();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty_acc[s]);
            }
            float b2;
            int i1;
            epi_resolve(b1, b2o, sv, sj, b2, i1);
            // merge the column groups of each row
            asm volatile("bar.sync 1, %0;" ::"r"(32 * TC_EPI_WARPS) : "memory");
            if (h > 0) {
                float *m = mrg + ((h - 1) * TC_M + rloc) * 3;
                m[0] = b1;
                m[1] = b2;
                m[2] = __int_as_float(i1);
            }
            asm volatile("bar.sync 1, %0;" ::"r"(32 * TC_EPI_WARPS) : "memory");
            if (h == 0 && row < I.n && ok) {
#pragma unroll
                for (int g = 1; g < TC_EPI_GROUPS; g++) {
                    const float *m = mrg + ((g - 1) * TC_M + rloc) * 3;
                    const float ob1 = m[0], ob2 = m[1];
                    const int oi1 = __float_as_int(m[2]);
                    // equal best values leave b2 == b1: the row is then
                    // flagged and decided in FP64, so the index is moot
                    float nb2;
                    if (ob1 < b1) {
                        nb2 = fminf(b1, fminf(b2, ob2));
                        b1 = ob1;
                        i1 = oi1;
                    } else {
                        nb2 = fminf(ob1, fminf(b2, ob2));
                    }
                    b2 = nb2;
                }
                const bool valid = i1 != 0x7FFFFFFF;
                I.labels[row] = valid ? i1 : -1;
                const bool sure = valid && (I.k == 1 || b2 - b1 > Wc);
                if (!sure) {
                    const unsigned long long qq = atomicAdd(A.n_flag, 1ull);
                    A.flag_rows[qq] = (int32_t)(I.row_base + row);
                    A.flag_m[qq] = valid ? b1 : __int_as_float(0x7fc00000);
                }
            }
            asm volatile("bar.sync 1, %0;" ::"r"(32 * TC_EPI_WARPS) : "memory");
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS) : "memory");
    }
}

// The BF16 pass over pairs of row tiles (one data set of many rows and centres).
// A centre tile is what bounds k_assign_tc at d = 128: per 128 x 256 tile the
// tensor core takes 9 k-steps of 128 cycles and reads 12 KB of shared memory for
// each, and the copy of the next centre tile writes 72 KB: 180 KB in 1,152 cycles
// is more than the 128 bytes a cycle that shared memory gives.  Here a centre
// tile serves two row tiles, row tile 0 into accumulator 0, row tile 1 into
// accumulator 1, so the copies write half as much per MMA (144 KB in 1,152
// cycles).  Both X stages hold the pair, so the next pair's first tile arrives
// while the last MMAs on the second one run; epilogue warps 2-5 own
// accumulator 0, 6-9 accumulator 1, each all 256 columns of its 32 rows (no
// merge).  10M x 128, k = 20,000: 34.4 ms, one row tile at a time 36.2 ms.
__global__ void __launch_bounds__(TC_THREADS, 1) k_assign_tc_pair(const __grid_constant__ TcArgs A) {
    extern __shared__ uint8_t smem_raw[];
    uint8_t *base = (uint8_t *)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
    uint8_t *sA0 = base, *sB0 = base + 2 * TC_A_STAGE;
    uint64_t *bars = (uint64_t *)(base + 2 * TC_A_STAGE + 2 * TC_B_STAGE);
    uint64_t *full_a = bars, *empty_a = bars + 2, *full_acc = bars + 4, *empty_acc = bars + 6;
    uint64_t *full_b = bars + 8, *empty_b = bars + 10, *done_bar = bars + 12;
    uint32_t *tmem_slot = (uint32_t *)(bars + 13);
    uint8_t *sOnes = base + 2 * TC_A_STAGE + 2 * TC_B_STAGE + TC_MISC;
    uint8_t *sX0 = sOnes + TC_M * 32;  // [2][TC_N * 32]
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; i++) {
            mbar_init(&full_a[i], 1);
            mbar_init(&empty_a[i], 1);
            mbar_init(&full_acc[i], 1);
            mbar_init(&empty_acc[i], TC_EPI_WARPS / 2);
            mbar_init(&full_b[i], 1);
            mbar_init(&empty_b[i], 1);
        }
        mbar_init(done_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    for (int e = threadIdx.x; e < TC_M * 32 / 4; e += blockDim.x)
        reinterpret_cast<uint32_t *>(sOnes)[e] = 0x3F803F80u;
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(su32(tmem_slot)),
                     "r"(TC_TMEM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_before();
    __syncthreads();
    fence_after();
    const uint32_t tmem = *tmem_slot;
    const TcInst &I = A.inst[0];
    const int nkb = I.Kp / TC_KB, ntc = I.ntiles_c, d = I.d;

    if (warp == 0) {
        // ------------------------------------------------ TMA producer
        if (lane == 0) {
            uint64_t ct = 0;
            uint32_t it = 0, issued_a[2] = {0, 0}, issued_b[2] = {0, 0};
            bool ok = true;
            for (int64_t u = blockIdx.x; u < A.nunits && ok; u += gridDim.x, it++) {
                for (int h = 0; h < 2; h++) {
                    if (!(ok = mbar_wait(&empty_a[h], (it & 1) ^ 1, A.err))) break;
                    mbar_expect_tx(&full_a[h], (uint32_t)(nkb * TC_M * 128));
                    // a second tile past the rows reads zeros
                    for (int kb = 0; kb < nkb; kb++)
                        tma_load_2d(su32(sA0 + h * TC_A_STAGE + kb * TC_M * 128), &I.tmA, kb * TC_KB,
                                    (int)(2 * u + h) * TC_M, &full_a[h]);
                    issued_a[h] = it + 1;
                }
                for (int c = 0; c < ntc && ok; c++, ct++) {
                    const int s = (int)(ct & 1);
                    const uint32_t uu = (uint32_t)(ct >> 1);
                    if (!(ok = mbar_wait(&empty_b[s], (uu & 1) ^ 1, A.err))) break;
                    mbar_expect_tx(&full_b[s], (uint32_t)(nkb * TC_N * 128 + TC_N * 32));
                    for (int kb = 0; kb < nkb; kb++)
                        tma_load_2d(su32(sB0 + s * TC_B_STAGE + kb * TC_N * 128), &I.tmB, kb * TC_KB, c * TC_N, &full_b[s]);
                    tma_load_2d(su32(sX0 + s * TC_N * 32), &I.tmX, 0, c * TC_N, &full_b[s]);
                    issued_b[s] = uu + 1;
                }
                if (!ok) break;
            }
            // drain: every copy this thread issued has landed
            for (int h = 0; h < 2; h++)
                if (issued_a[h]) mbar_wait(&full_a[h], (issued_a[h] - 1) & 1, A.err, true);
            for (int s = 0; s < 2; s++)
                if (issued_b[s]) mbar_wait(&full_b[s], (issued_b[s] - 1) & 1, A.err, true);
        }
        __syncwarp();
    } else if (warp == 1) {
        // ------------------------------------------------ MMA issuer
        if (lane == 0) {
            uint64_t ct = 0;
            uint32_t it = 0;
            bool ok = true;
            const uint32_t idesc = idesc_bf16(TC_M, TC_N);
            for (int64_t u = blockIdx.x; u < A.nunits && ok; u += gridDim.x, it++) {
                for (int c = 0; c < ntc && ok; c++, ct++) {
                    const int s = (int)(ct & 1);
                    if (!(ok = mbar_wait(&full_b[s], (uint32_t)(ct >> 1) & 1, A.err))) break;
                    for (int h = 0; h < 2; h++) {
                        if (!(ok = mbar_wait(&empty_acc[h], ((uint32_t)ct & 1) ^ 1, A.err))) break;
                        if (c == 0 && !(ok = mbar_wait(&full_a[h], it & 1, A.err))) break;
                        fence_after();
                        const uint32_t dtm = tmem + (uint32_t)(h * TC_N);
                        for (int kb = 0; kb < nkb; kb++) {
                            const uint64_t da = sdesc(su32(sA0 + h * TC_A_STAGE + kb * TC_M * 128));
                            const uint64_t db = sdesc(su32(sB0 + s * TC_B_STAGE + kb * TC_N * 128));
#pragma unroll
                            for (int ks = 0; ks < TC_KB / 16; ks++) {
                                if (kb * TC_KB + ks * 16 >= d) break;  // zeros from here on
                                mma_bf16(dtm, da + 2 * ks, db + 2 * ks, idesc, (kb | ks) != 0);
                            }
                        }
                        // + |c|^2
                        mma_bf16(dtm, sdesc32(su32(sOnes)), sdesc32(su32(sX0 + s * TC_N * 32)), idesc, 1);
                        mma_commit(&full_acc[h]);
                        if (c + 1 == ntc) mma_commit(&empty_a[h]);
                    }
                    if (!ok) break;
                    mma_commit(&empty_b[s]);
                }
            }
            // drain: all MMAs this thread issued have completed
            mma_commit(done_bar);
            mbar_wait(done_bar, 0, A.err, true);
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ epilogue
        const int q = warp & 3;         // TMEM lane quarter this warp may access
        const int h = (warp - 2) >> 2;  // its accumulator
        const uint32_t tbase = tmem + (uint32_t)(h * TC_N) + ((uint32_t)(32 * q) << 16);
        const float cmax = sqrtf(__uint_as_float(*I.cmax_bits)) * (1.f + 1e-5f);
        uint64_t ct = 0;
        bool ok = true;
        for (int64_t u = blockIdx.x; u < A.nunits; u += gridDim.x) {
            const int64_t row = (2 * u + h) * TC_M + 32 * q + lane;
            const float xn = row < I.n ? I.xnorm[row] : 0.f;
            const float Wc = 2.f * window_bf16(xn, cmax, I.d) * (1.f + 1e-6f);
            float b1 = FLT_MAX, b2o = FLT_MAX, sv[32];
            int64_t sj = -1;
            for (int c = 0; c < ntc; c++, ct++) {
                int w_ok = 0;
                if (lane == 0 && ok) w_ok = mbar_wait(&full_acc[h], (uint32_t)ct & 1, A.err);
                w_ok = __shfl_sync(0xffffffffu, w_ok, 0);
                ok = ok && w_ok;
                if (ok) {
                    fence_after();
                    epi_tile<TC_N / 32>(tbase, (int64_t)c * TC_N, b1, b2o, sv, sj);
                    fence_before();
                }
                __syncwarp();
                if (lane == 0) mbar_arrive(&empty_acc[h]);
            }
            float b2;
            int i1;
            epi_resolve(b1, b2o, sv, sj, b2, i1);
            if (row < I.n && ok) {
                const bool valid = i1 != 0x7FFFFFFF;
                I.labels[row] = valid ? i1 : -1;
                if (!(valid && (I.k == 1 || b2 - b1 > Wc))) {
                    const unsigned long long qq = atomicAdd(A.n_flag, 1ull);
                    A.flag_rows[qq] = (int32_t)(I.row_base + row);
                    A.flag_m[qq] = valid ? b1 : __int_as_float(0x7fc00000);
                }
            }
        }
    }
    fence_before();
    __syncthreads();
    if (warp == 0) {
        fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(TC_TMEM_COLS) : "memory");
    }
}

// X -> BF16 K-major [n][Kp] (zero padded) and an upper bound of |x| per row;
// xnorm is global.  One read and one write of memory bound it.  With 16-byte
// rows Kp / 4 lanes take a row, four consecutive columns each (float4 loads, 8-byte
// stores).  In a batch a warp takes a stretch of rows, four such loads in flight
// per lane, 4 rows of 128 columns or 8 of 64 (33.75M rows: 5.7 ms with a row at a
// time, now 3.8); one instance's rows are strided over the warps, a row each, so
// that all of them work on one stretch of memory (10M x 128: 1.26 ms; in groups of
// four 1.8, with the instance's fields read again for every row 1.52).
constexpr int XB_U = 4;
template <int U>
__device__ __forceinline__ void x_rows_to_bf16(const TcXPrep &P, int64_t i0, int64_t i1, float *__restrict__ xnorm) {
    const int lane = threadIdx.x & 31;
    const int lpr = P.Kp >> 2, rps = 32 / lpr;  // lanes per row (16 or 32), rows per step
    const int t = 4 * (lane & (lpr - 1)), sub = lane / lpr;
    const int W = P.split ? 2 * P.Kp : P.Kp;
    float4 v[U];
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int64_t i = i0 + u * rps + sub;
        v[u] = i < i1 && t < P.d ? *reinterpret_cast<const float4 *>(P.x + i * P.ldx + t) : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int u = 0; u < U; u++) {
        const int64_t i = i0 + u * rps + sub;
        const __nv_bfloat162 h01 = __floats2bfloat162_rn(v[u].x, v[u].y), h23 = __floats2bfloat162_rn(v[u].z, v[u].w);
        if (i < i1) {
            __nv_bfloat16 *hb = P.xb + i * W;
            uint2 hv;
            hv.x = *reinterpret_cast<const uint32_t *>(&h01);
            hv.y = *reinterpret_cast<const uint32_t *>(&h23);
            *reinterpret_cast<uint2 *>(hb + t) = hv;
            if (P.split) {
                const float2 f01 = __bfloat1622float2(h01), f23 = __bfloat1622float2(h23);
                const __nv_bfloat162 l01 = __floats2bfloat162_rn(v[u].x - f01.x, v[u].y - f01.y);  // differences exact
                const __nv_bfloat162 l23 = __floats2bfloat162_rn(v[u].z - f23.x, v[u].w - f23.y);
                uint2 lv;
                lv.x = *reinterpret_cast<const uint32_t *>(&l01);
                lv.y = *reinterpret_cast<const uint32_t *>(&l23);
                *reinterpret_cast<uint2 *>(hb + P.Kp + t) = lv;
            }
        }
        float s = fmaf(v[u].x, v[u].x, fmaf(v[u].y, v[u].y, fmaf(v[u].z, v[u].z, v[u].w * v[u].w)));
        for (int o = lpr >> 1; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((lane & (lpr - 1)) == 0 && i < i1) xnorm[i] = sqrtf(s) * (1.f + 1.0e-3f);
    }
}
// a row of any alignment, by a warp
__device__ __forceinline__ void x_row_to_bf16(const TcXPrep &P, int64_t i, float *__restrict__ xnorm) {
    const int lane = threadIdx.x & 31;
    const float *xr = P.x + i * P.ldx;
    __nv_bfloat16 *hb = P.xb + i * (P.split ? 2 * P.Kp : P.Kp);
    float s = 0.f;
    for (int t = lane; t < P.Kp; t += 32) {
        const float v = t < P.d ? xr[t] : 0.f;
        const __nv_bfloat16 h = __float2bfloat16_rn(v);
        hb[t] = h;
        if (P.split) hb[P.Kp + t] = __float2bfloat16_rn(v - __bfloat162float(h));  // v - h exact
        s = fmaf(v, v, s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) xnorm[i] = sqrtf(s) * (1.f + 1.0e-3f);
}
__device__ __forceinline__ bool x_vec(const TcXPrep &P) {
    return ((P.ldx & 3) == 0) && ((P.d & 3) == 0) && (((uintptr_t)P.x & 15) == 0);
}
__global__ void k_x_to_bf16_one(const TcXPrep *__restrict__ X, int64_t n, float *__restrict__ xnorm) {
    const TcXPrep P = X[0];
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    if (x_vec(P)) {
        const int64_t rows = 128 / P.Kp;  // a row of 128 columns or two of 64
        for (int64_t i = warp * rows; i < n; i += nw * rows) x_rows_to_bf16<1>(P, i, n, xnorm);
    } else {
        for (int64_t i = warp; i < n; i += nw) x_row_to_bf16(P, i, xnorm);
    }
}
__global__ void k_x_to_bf16_batch(const TcXPrep *__restrict__ X, const int64_t *__restrict__ row_off, int count,
                                  int64_t N, float *__restrict__ xnorm) {
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t per = (N + nw - 1) / nw, rend = min(N, (warp + 1) * per);
    for (int64_t r = warp * per; r < rend;) {  // the stretch, in pieces that end with their instance
        const int ii = find_inst(row_off, count, r);
        const TcXPrep P = X[ii];
        const int64_t base = row_off[ii], iend = min(rend, row_off[ii + 1]) - base;
        int64_t i = r - base;
        r = base + iend;
        if (x_vec(P)) {
            for (; i < iend; i += XB_U * (128 / P.Kp)) x_rows_to_bf16<XB_U>(P, i, iend, xnorm + base);
        } else {
            for (; i < iend; i++) x_row_to_bf16(P, i, xnorm + base);
        }
    }
}

// centres -> BF16 [kpad][Kp], |c|^2 (+inf for padding) and the max of |c|^2 over
// real centres; centre e is global, padded ones included, of instance
// find_inst(kpad_off, e).  The warps take them as in the FP32 copy (assign.cu,
// centre_prep), and for the same reason: 1M x 32 takes 419 us, 1,479 with a warp
// per centre, 200,000 x 128 170 us, 440; with a thread per centre, each store two
// bytes of another row, 2,048 split ones took 66 us, now 7.
__global__ void k_c_to_bf16(const TcCPrep *__restrict__ C, const int64_t *__restrict__ kpad_off, int count,
                            int64_t total, CentreWarp W) {
    const int lane = threadIdx.x & 31, per = W.per_step();
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * W.centres() < total; w += nw) {
        const int64_t e0 = w * W.centres();
        double mine = 0.0;
        for (int st = 0; st < W.steps; st++) {
            const int64_t e = e0 + per * st + lane / W.lanes;
            double s = 0.0;
            if (e < total) {
                const int ii = find_inst(kpad_off, count, e);
                const TcCPrep &P = C[ii];
                const int64_t j = e - kpad_off[ii];
                const int Kp = P.Kp;
                const bool split = P.split;
                const int d = j < P.k ? P.d : 0;
                const double *c = P.c + j * P.d;
                __nv_bfloat16 *cb = P.cb + j * (split ? 2 * Kp : Kp);
#pragma unroll 4
                for (int t = 2 * (lane & (W.lanes - 1)); t < Kp; t += 2 * W.lanes) {
                    // -2 c: scaling by a power of two is exact in BF16
                    const double v0 = t < d ? c[t] : 0.0, v1 = t + 1 < d ? c[t + 1] : 0.0;
                    const double a0 = -2.0 * v0, a1 = -2.0 * v1;
                    __nv_bfloat162 h;
                    h.x = __double2bfloat16(a0);
                    h.y = __double2bfloat16(a1);
                    *reinterpret_cast<__nv_bfloat162 *>(cb + t) = h;
                    if (split) {
                        __nv_bfloat162 l;
                        l.x = __double2bfloat16(a0 - (double)__bfloat162float(h.x));  // exact
                        l.y = __double2bfloat16(a1 - (double)__bfloat162float(h.y));
                        *reinterpret_cast<__nv_bfloat162 *>(cb + Kp + t) = l;
                    }
                    s += v0 * v0;
                    s += v1 * v1;
                }
            }
            for (int o = 1; o < W.lanes; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            s = __shfl_sync(0xffffffffu, s, W.lanes * (lane & (per - 1)));
            if (lane / per == st) mine = s;
        }
        const int64_t e = e0 + lane;
        unsigned bits = 0;
        unsigned *most = nullptr;
        if (lane < W.centres() && e < total) {
            const int ii = find_inst(kpad_off, count, e);
            const TcCPrep &P = C[ii];
            const int64_t j = e - kpad_off[ii];
            // |c|^2 = hi + mid + lo in BF16 (within 2^-24 |c|^2); padding: +inf,
            // which never wins
            uint32_t hm = 0x7F80u, l = 0u;
            if (j < P.k) {
                const __nv_bfloat16 h = __double2bfloat16(mine);
                const double r1 = mine - (double)__bfloat162float(h);
                const __nv_bfloat16 m = __double2bfloat16(r1);
                hm = (uint32_t)__bfloat16_as_ushort(h) | (uint32_t)__bfloat16_as_ushort(m) << 16;
                l = __bfloat16_as_ushort(__double2bfloat16(r1 - (double)__bfloat162float(m)));
                bits = __float_as_uint((float)mine);  // non-negative floats order as uints
                most = P.cmax_bits;
            }
            uint4 *x = reinterpret_cast<uint4 *>(P.cbx + j * 16);
            x[0] = make_uint4(hm, l, 0u, 0u);
            x[1] = make_uint4(0u, 0u, 0u, 0u);
            P.cn[j] = j < P.k ? (float)mine : __int_as_float(0x7f800000);
        }
        max_by_warp(most, bits);
    }
}

constexpr int TC_TILES[3] = {64, 128, 256};

}  // namespace

struct TcPlan::Impl {
    std::vector<TcInst> inst;      // host copy (tensor maps for the chosen N)
    std::vector<TcXPrep> xp;
    std::vector<TcCPrep> cp;
    std::vector<int64_t> kpad_off;
};

namespace {

template <class T>
geek_status plan_alloc(geek_ctx *ctx, Scratch *scr, std::vector<void *> &owned, T **p, size_t count) {
    if (scr) return scr->alloc(p, count);
    if (alloc_injected_failure(ctx))
        return set_error(ctx, GEEK_ERR_NOMEM, "device allocation of %zu bytes failed (injected)", count * sizeof(T));
    void *q = nullptr;
    cudaError_t e = cudaMalloc(&q, std::max<size_t>(count * sizeof(T), 16));
    if (e != cudaSuccess) {
        cudaGetLastError();
        return set_error(ctx, GEEK_ERR_NOMEM, "device allocation of %zu bytes failed", count * sizeof(T));
    }
    owned.push_back(q);
    *p = (T *)q;
    return GEEK_OK;
}

// TcInst of instance i for tile width N (tensor maps re-encoded)
geek_status make_inst(geek_ctx *ctx, const TcPlan &P, int i, int N, TcInst *out) {
    const TcPlanInst &I = P.desc[i];
    const int Kp = I.d <= 64 ? 64 : 128;
    TcInst T;
    memset(&T, 0, sizeof T);
    const TcXPrep &xp = P.impl->xp[i];
    const TcCPrep &cp = P.impl->cp[i];
    const int Kst = I.split ? 2 * Kp : Kp;  // stored columns
    if (I.split && N * Kp > 8192 && P.count != 1)
        return set_error(ctx, GEEK_ERR_INVALID, "split-BF16 tiles of a batch need N * Kp <= 8192 (N %d, Kp %d)", N, Kp);
    if (I.n > 0) GK_TRY(encode_bf16_2d(ctx, &T.tmA, xp.xb, Kst, I.n, TC_KB, TC_M));
    if (I.k > 0) GK_TRY(encode_bf16_2d(ctx, &T.tmB, cp.cb, Kst, cp.kpad, TC_KB, N));
    if (I.k > 0) GK_TRY(encode_bf16_2d(ctx, &T.tmX, cp.cbx, 16, cp.kpad, 16, N, CU_TENSOR_MAP_SWIZZLE_32B));
    T.xnorm = P.xnorm + I.row_base;
    T.cmax_bits = cp.cmax_bits;
    T.labels = I.labels;
    T.n = I.n;
    T.k = I.k;
    T.row_base = I.row_base;
    T.ntiles_c = (int)ceil_div(I.k, N);
    T.Kp = Kp;
    T.d = I.d;
    T.N = N;
    T.split = I.split;
    *out = T;
    return GEEK_OK;
}

// units of the listed instances in one mode (split or not), longest first
// (LPT order over the CTAs)
void make_units(const TcPlan &P, const std::vector<int> &which, int split, std::vector<int2> &units) {
    std::vector<std::pair<int64_t, int>> cost;
    for (int i : which) {
        const TcInst &T = P.impl->inst[i];
        if (T.n <= 0 || T.k <= 0 || P.desc[i].split != split) continue;
        cost.push_back({(int64_t)T.ntiles_c * T.N * T.Kp * (split ? 3 : 1) + 2048, i});
    }
    std::stable_sort(cost.begin(), cost.end(), [](const std::pair<int64_t, int> &a, const std::pair<int64_t, int> &b) {
        return a.first > b.first;
    });
    units.clear();
    for (auto &c : cost) {
        const int64_t nt = ceil_div(P.impl->inst[c.second].n, TC_M);
        for (int64_t r = 0; r < nt; r++) units.push_back(make_int2(c.second, (int)r));
    }
}

size_t tc_smem() {
    static_assert(32 * 8 + (TC_EPI_GROUPS - 1) * TC_M * 3 * 4 <= TC_MISC, "misc region too small");
    // tile stages + barriers / TMEM slot / merge buffer + ones block + two
    // |c|^2 stages + alignment
    return 1024 + 2 * (size_t)TC_A_STAGE + 2 * (size_t)TC_B_STAGE + TC_MISC + TC_M * 32 + 2 * TC_N * 32;
}

}  // namespace

int tc_tile_candidates(const int **tiles) {
    *tiles = TC_TILES;
    return 3;
}

geek_status tc_plan_build(geek_ctx *ctx, Scratch *scr, const std::vector<TcPlanInst> &desc, TcPlan *P,
                          cudaStream_t st) {
    P->impl = new TcPlan::Impl();
    P->desc = desc;
    const int count = (int)desc.size();
    P->count = count;
    auto &im = *P->impl;
    std::vector<int64_t> row_off(count + 1, 0);
    im.kpad_off.assign(count + 1, 0);
    int64_t xb_total = 0, cb_total = 0;
    for (int i = 0; i < count; i++) {
        const TcPlanInst &I = desc[i];
        if (I.d > TC_KP_MAX || I.d <= 0)
            return set_error(ctx, GEEK_ERR_UNSUPPORTED, "BF16 tensor-core assignment supports 1 <= d <= 128");
        if (I.N != 64 && I.N != 128 && I.N != 256) return set_error(ctx, GEEK_ERR_INVALID, "tile N must be 64/128/256");
        const int Kp = I.d <= 64 ? 64 : 128;
        // room for the split layout whenever a plan may switch modes
        const int Kst = (I.split || P->allow_split) ? 2 * Kp : Kp;
        row_off[i + 1] = row_off[i] + I.n;
        // padding to a multiple of 256 serves every tile width
        im.kpad_off[i + 1] = im.kpad_off[i] + ceil_div(I.k, TC_N) * TC_N;
        xb_total += I.n * Kst;
        cb_total += ceil_div(I.k, TC_N) * TC_N * Kst;
    }
    P->N_total = row_off[count];
    P->kpad_total = im.kpad_off[count];
    auto &own = P->owned;
    __nv_bfloat16 *xb, *cb, *cbx;
    float *cn;
    unsigned *cmax_bits;
    if (P->x_done) xb = P->x_done->xb;
    else GK_TRY(plan_alloc(ctx, scr, own, &xb, (size_t)std::max<int64_t>(xb_total, 1)));
    GK_TRY(plan_alloc(ctx, scr, own, &cb, (size_t)std::max<int64_t>(cb_total, 1)));
    GK_TRY(plan_alloc(ctx, scr, own, &cbx, (size_t)std::max<int64_t>(im.kpad_off[count] * 16, 1)));
    if (P->x_done) P->xnorm = P->x_done->xnorm;
    else GK_TRY(plan_alloc(ctx, scr, own, &P->xnorm, (size_t)std::max<int64_t>(P->N_total, 1)));
    GK_TRY(plan_alloc(ctx, scr, own, &cn, (size_t)std::max<int64_t>(P->kpad_total, 1)));
    GK_TRY(plan_alloc(ctx, scr, own, &cmax_bits, (size_t)count));
    GK_TRY(plan_alloc(ctx, scr, own, &P->row_off, (size_t)count + 1));
    GK_TRY(plan_alloc(ctx, scr, own, &P->kpad_off_dev, (size_t)count + 1));
    GK_TRY(plan_alloc(ctx, scr, own, &P->xprep, (size_t)count));
    GK_TRY(plan_alloc(ctx, scr, own, &P->cprep, (size_t)count));
    GK_TRY(plan_alloc(ctx, scr, own, &P->inst, (size_t)count));
    GK_TRY(plan_alloc(ctx, scr, own, &P->err, 1));
    P->cmax_bits = cmax_bits;
    im.xp.resize(count);
    im.cp.resize(count);
    int64_t xo = 0, co = 0;
    for (int i = 0; i < count; i++) {
        const TcPlanInst &I = desc[i];
        const int Kp = I.d <= 64 ? 64 : 128;
        const int Kst = (I.split || P->allow_split) ? 2 * Kp : Kp;
        im.xp[i] = TcXPrep{I.x, I.ldx, I.d, Kp, I.split, xb + xo};
        const int64_t kpad = im.kpad_off[i + 1] - im.kpad_off[i];
        im.cp[i] = TcCPrep{I.centres, I.k, kpad, I.d, Kp, I.split, cb + co, cbx + im.kpad_off[i] * 16,
                           cn + im.kpad_off[i], cmax_bits + i};
        xo += I.n * Kst;
        co += kpad * Kst;
    }
    im.inst.resize(count);
    for (int i = 0; i < count; i++) GK_TRY(make_inst(ctx, *P, i, desc[i].N, &im.inst[i]));
    GK_TRY(plan_alloc(ctx, scr, own, &P->units, (size_t)std::max<int64_t>(ceil_div(P->N_total, TC_M) + count, 1)));
    GK_CUDA(ctx, cudaMemcpyAsync(P->row_off, row_off.data(), sizeof(int64_t) * (count + 1), cudaMemcpyHostToDevice, st));
    GK_CUDA(ctx, cudaMemcpyAsync(P->kpad_off_dev, im.kpad_off.data(), sizeof(int64_t) * (count + 1),
                                 cudaMemcpyHostToDevice, st));
    GK_TRY(tc_plan_upload(ctx, P, st));
    for (const void *fn : {(const void *)k_assign_tc<false, false>, (const void *)k_assign_tc<true, false>,
                           (const void *)k_assign_tc<false, true>, (const void *)k_assign_tc<true, true>,
                           (const void *)k_assign_tc_pair})
        GK_CUDA(ctx, cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)tc_smem()));
    return GEEK_OK;
}

// Uploads the descriptors and unit lists of the current modes and tiles:
// units[0, nunits) run in BF16, units[nunits, nunits + nunits_x3) in
// split-BF16.
geek_status tc_plan_upload(geek_ctx *ctx, TcPlan *P, cudaStream_t st) {
    auto &im = *P->impl;
    const int count = P->count;
    for (int i = 0; i < count; i++) {
        im.xp[i].split = P->desc[i].split;
        im.cp[i].split = P->desc[i].split;
    }
    std::vector<int> all(count);
    for (int i = 0; i < count; i++) all[i] = i;
    std::vector<int2> u0, u1;
    make_units(*P, all, 0, u0);
    make_units(*P, all, 1, u1);
    P->nunits = (int64_t)u0.size();
    P->nunits_x3 = (int64_t)u1.size();
    u0.insert(u0.end(), u1.begin(), u1.end());
    GK_CUDA(ctx, cudaMemcpyAsync(P->xprep, im.xp.data(), sizeof(TcXPrep) * count, cudaMemcpyHostToDevice, st));
    GK_CUDA(ctx, cudaMemcpyAsync(P->cprep, im.cp.data(), sizeof(TcCPrep) * count, cudaMemcpyHostToDevice, st));
    GK_CUDA(ctx, cudaMemcpyAsync(P->inst, im.inst.data(), sizeof(TcInst) * count, cudaMemcpyHostToDevice, st));
    if (!u0.empty())
        GK_CUDA(ctx, cudaMemcpyAsync(P->units, u0.data(), sizeof(int2) * u0.size(), cudaMemcpyHostToDevice, st));
    // the host vectors are pageable: the copies have read them on return
    return GEEK_OK;
}

// Conversions of X and the centres (BF16 or split-BF16 pairs, norms, the
// max of |c|^2).  No host synchronisation.
geek_status tc_plan_convert(geek_ctx *ctx, const TcPlan &P, cudaStream_t st) {
    const int count = P.count;
    GK_CUDA(ctx, cudaMemsetAsync(P.err, 0, sizeof(int), st));
    GK_CUDA(ctx, cudaMemsetAsync(P.cmax_bits, 0, sizeof(unsigned) * count, st));
    if (P.N_total > 0 && !P.x_done) {
        GK_COUNT();
        const int g = grid_for(P.N_total * 32, 256, ctx->num_sms);
        if (count == 1) k_x_to_bf16_one<<<g, 256, 0, st>>>(P.xprep, P.N_total, P.xnorm);
        else k_x_to_bf16_batch<<<g, 256, 0, st>>>(P.xprep, P.row_off, count, P.N_total, P.xnorm);
    }
    if (P.kpad_total > 0) {
        GK_COUNT();
        const CentreWarp cw = centre_warp(ctx, P.kpad_total);
        k_c_to_bf16<<<grid_for(ceil_div(P.kpad_total, cw.centres()) * 32, 128, ctx->num_sms), 128, 0, st>>>(
            P.cprep, P.kpad_off_dev, count, P.kpad_total, cw);
    }
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

namespace {

// The rings for the instances of one mode in a launch: log2 of the centre
// ring's stages (2 .. 8) and of the |c|^2 ring's.  The widest tile among them
// fixes the stage size, and the ring's bytes are cut into as many stages as fit;
// both regions bound the count (the |c|^2 rows, N x 32 bytes a tile, have 2 TC_N
// * 32).  A tile wider than half the ring (one split instance, N = 256, Kp =
// 128) goes through in 64-column parts, four stages, and its |c|^2 rows take
// turns in two: a part's stage comes free only after every part before it.
struct Rings {
    int ns, nx, na;
};
Rings ring_lg(const TcPlan &P, const std::vector<int> *which, int split) {
    int64_t mx = 0, nmax = 0;
    auto consider = [&](int i) {
        const TcPlanInst &I = P.desc[i];
        if ((I.split != 0) != (split != 0)) return;
        const int64_t Kp = I.d <= 64 ? 64 : 128;
        mx = std::max<int64_t>(mx, (int64_t)I.N * Kp * 2 * (split ? 2 : 1));
        nmax = std::max<int64_t>(nmax, (int64_t)I.N);
    };
    if (which)
        for (int i : *which) consider(i);
    else
        for (int i = 0; i < P.count; i++) consider(i);
    // split tiles of N Kp <= 8192: four X stages, the centre ring half as large
    const int lg_na = split && mx <= TC_B_STAGE / 2 ? 2 : 1;
    const int64_t ring = 2 * (int64_t)TC_B_STAGE - ((1 << lg_na) - 2) * (int64_t)TC_A_STAGE;
    if (mx > ring / 2) return Rings{2, 1, lg_na};
    int lg = 1;
    const int64_t xring = 2 * (int64_t)TC_N * 32;
    while (lg < 3 && mx > 0 && (ring >> (lg + 1)) >= mx && (xring >> (lg + 1)) >= nmax * 32) lg++;
    return Rings{lg, lg, lg_na};
}

// Pairs of row tiles: one BF16 data set of 256-wide tiles, several centre tiles per
// pair (the next pair's rows are loaded only at the end of this one), four pairs
// or more per SM.  Pairs come out even on the SMs less often than single tiles:
// what the longer last round costs, 2 ceil(pairs / SMs) against ceil(tiles / SMs),
// must stay below what a pair saves, 1 % and a part that shrinks with the centres
// (the ends of a row tile, twice as large a share with d <= 64).  Times against one
// tile at a time, k = 2,048 / 4,000 / 20,000 / 100,000: with even rounds (n =
// 311,296) d = 64: 0.89 / 0.92 / 0.97 / 0.99, d = 128: 0.94 / 1.00 / 0.97 / 0.89; with
// 22 for 21 (n = 400,000) d = 64: 0.92 / 0.95 / 1.02 / 1.04, d = 128: 0.99 / 1.04 / 1.02;
// with 10 for 9 (n = 156,000) d = 64: 0.97 / 1.02 / 1.07 / 1.10, d = 128: 1.05 / 1.10 /
// 1.09 / 1.03.
bool pairs_pay(const TcPlanInst &I, int num_sms) {
    const int64_t pairs = ceil_div(I.n, 2 * TC_M), tiles_c = ceil_div(I.k, TC_N);
    if (I.split || I.N != TC_N || pairs < 4 * (int64_t)num_sms || tiles_c < 8) return false;
    const double rounds = (double)ceil_div(I.n, (int64_t)TC_M * num_sms);
    return 2.0 * (double)ceil_div(pairs, num_sms) <= rounds * (1.01 + (I.d <= 64 ? 1.0 : 0.4) / (double)tiles_c);
}

geek_status launch_units(geek_ctx *ctx, const TcInst *inst, const int2 *units, int64_t n0, int64_t n1,
                         int32_t *flag_rows, float *flag_m, unsigned long long *n_flag, int *err, double work,
                         Rings r0, Rings r1, cudaStream_t st) {
    TcArgs A{};
    A.inst = inst;
    A.flag_rows = flag_rows;
    A.flag_m = flag_m;
    A.n_flag = n_flag;
    A.err = err;
    EvTimer tk(ctx, "kernel.assign_tc", st);
    tk.work = work;
    if (n0 > 0) {
        A.units = units;
        A.nunits = n0;
        A.lg_ns = r0.ns;
        A.lg_nx = r0.nx;
        A.lg_na = r0.na;
        GK_COUNT();
        k_assign_tc<false, false><<<(int)std::min<int64_t>(n0, ctx->num_sms), TC_THREADS, tc_smem(), st>>>(A);
    }
    if (n1 > 0) {
        A.units = units + n0;
        A.nunits = n1;
        A.lg_ns = r1.ns;
        A.lg_nx = r1.nx;
        A.lg_na = r1.na;
        GK_COUNT();
        k_assign_tc<true, false><<<(int)std::min<int64_t>(n1, ctx->num_sms), TC_THREADS, tc_smem(), st>>>(A);
    }
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

}  // namespace

// The persistent tcgen05 passes (BF16 units, then split-BF16 units) after
// tc_plan_convert; flagged rows are appended to flag_rows / n_flag (zeroed
// by the caller).
geek_status tc_plan_launch(geek_ctx *ctx, const TcPlan &P, int32_t *flag_rows, float *flag_m,
                           unsigned long long *n_flag, cudaStream_t st) {
    double work = 0.0;
    for (const TcPlanInst &I : P.desc) work += 2.0 * (double)I.n * (double)I.k * (double)I.d;
    if (P.count == 1 && pairs_pay(P.desc[0], ctx->num_sms)) {
        TcArgs A{};
        A.inst = P.inst;
        A.nunits = ceil_div(P.desc[0].n, 2 * TC_M);
        A.flag_rows = flag_rows;
        A.flag_m = flag_m;
        A.n_flag = n_flag;
        A.err = P.err;
        EvTimer tk(ctx, "kernel.assign_tc", st);
        tk.work = work;
        GK_COUNT();
        k_assign_tc_pair<<<ctx->num_sms, TC_THREADS, tc_smem(), st>>>(A);
        GK_LAUNCH(ctx);
        return GEEK_OK;
    }
    return launch_units(ctx, P.inst, P.units, P.nunits, P.nunits_x3, flag_rows, flag_m, n_flag, P.err, work,
                        ring_lg(P, nullptr, 0), ring_lg(P, nullptr, 1), st);
}

geek_status tc_plan_enqueue(geek_ctx *ctx, const TcPlan &P, int32_t *flag_rows, float *flag_m,
                            unsigned long long *n_flag, cudaStream_t st) {
    GK_TRY(tc_plan_convert(ctx, P, st));
    return tc_plan_launch(ctx, P, flag_rows, flag_m, n_flag, st);
}

// Sets every instance's tile width and mode (descriptors re-encoded, units
// rebuilt).  The next tc_plan_convert writes the matching layouts.
geek_status tc_plan_set_modes(geek_ctx *ctx, TcPlan *P, const std::vector<int> &N, const std::vector<int> &split,
                              cudaStream_t st) {
    for (int i = 0; i < P->count; i++) {
        if (split[i] && !P->allow_split && !P->desc[i].split)
            return set_error(ctx, GEEK_ERR_INVALID, "plan was built without room for split-BF16");
        P->desc[i].N = N[i];
        P->desc[i].split = split[i];
        GK_TRY(make_inst(ctx, *P, i, N[i], &P->impl->inst[i]));
    }
    return tc_plan_upload(ctx, P, st);
}

// Launches the tcgen05 pass over the units of `which` only, with tile width
// N and mode `split` for those instances (their layouts must match: run
// tc_plan_convert after tc_plan_set_modes).  Uses the plan's scratch
// descriptor table; writes labels and flags of those rows.  No host sync.
geek_status tc_plan_launch_subset(geek_ctx *ctx, TcPlan *P, const std::vector<int> &which, int32_t *flag_rows,
                                  float *flag_m, unsigned long long *n_flag, cudaStream_t st) {
    auto &im = *P->impl;
    std::vector<int2> u0, u1;
    make_units(*P, which, 0, u0);
    make_units(*P, which, 1, u1);
    const int64_t n0 = (int64_t)u0.size(), n1 = (int64_t)u1.size();
    u0.insert(u0.end(), u1.begin(), u1.end());
    if (u0.empty()) return GEEK_OK;
    if (!P->tune_units || P->tune_cap < (int64_t)u0.size()) {
        if (P->tune_units) cudaFree(P->tune_units);
        P->tune_units = nullptr;
        P->tune_cap = 0;
        if (cudaMalloc((void **)&P->tune_units, sizeof(int2) * u0.size()) != cudaSuccess) {
            cudaGetLastError();
            return set_error(ctx, GEEK_ERR_NOMEM, "autotune unit list");
        }
        P->tune_cap = (int64_t)u0.size();
    }
    GK_CUDA(ctx, cudaMemcpyAsync(P->tune_units, u0.data(), sizeof(int2) * u0.size(), cudaMemcpyHostToDevice, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));  // u0 is pageable and about to go out of scope
    (void)im;
    return launch_units(ctx, P->inst, P->tune_units, n0, n1, flag_rows, flag_m, n_flag, P->err, 0.0,
                        ring_lg(*P, &which, 0), ring_lg(*P, &which, 1), st);
}

geek_status tc_plan_check(geek_ctx *ctx, const TcPlan &P, cudaStream_t st) {
    int h_err = 0;
    GK_CUDA(ctx, cudaMemcpyAsync(&h_err, P.err, sizeof h_err, cudaMemcpyDeviceToHost, st));
    GK_CUDA(ctx, cudaStreamSynchronize(st));
    if (h_err) return set_error(ctx, (geek_status)h_err, "tensor-core assignment: a pipeline wait timed out");
    return GEEK_OK;
}

void tc_plan_free(TcPlan *P) {
    for (void *p : P->owned) cudaFree(p);
    P->owned.clear();
    if (P->tune_units) cudaFree(P->tune_units);
    P->tune_units = nullptr;
    P->tune_cap = 0;
    delete P->impl;
    P->impl = nullptr;
}

geek_status tc_x_alloc(geek_ctx *ctx, Scratch &scr, int64_t n, int d, int split, TcX *X) {
    const int Kp = d <= 64 ? 64 : 128;
    GK_TRY(scr.alloc(&X->xb, (size_t)n * Kp * (split ? 2 : 1)));
    GK_TRY(scr.alloc(&X->xnorm, (size_t)n));
    return scr.alloc(&X->prep, 1);
}

geek_status tc_x_convert(geek_ctx *ctx, const float *x, int64_t ldx, int64_t n, int d, int split, const TcX &X,
                         cudaStream_t st) {
    const TcXPrep p{x, ldx, d, d <= 64 ? 64 : 128, split, X.xb};
    GK_CUDA(ctx, cudaMemcpyAsync(X.prep, &p, sizeof p, cudaMemcpyHostToDevice, st));  // pageable: read on return
    GK_COUNT();
    k_x_to_bf16_one<<<grid_for(n * 32, 256, ctx->num_sms), 256, 0, st>>>(X.prep, n, X.xnorm);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

// BF16 (split = 0) or split-BF16 (split = 1) tcgen05 pass of one data set:
// labels for every object, flagged rows appended to flag_rows / flag_m / n_flag
// for the exact decision, which may use the plan P (buffers in scr); the caller
// ends it with tc_plan_check.  d <= 128.
geek_status assign_tc_bf16(geek_ctx *ctx, Scratch &scr, const float *x, int64_t ldx, int64_t n, int d,
                           const double *centres, int64_t k, int split, int32_t *labels, int32_t *flag_rows,
                           float *flag_m, unsigned long long *n_flag, TcPlan *P, cudaStream_t st) {
    if (d > 128) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "BF16 tensor-core assignment supports d <= 128");
    std::vector<TcPlanInst> one(1);
    // the widest tiles (128-wide ones read the X tile from shared memory twice as
    // often per flop and measured ~60% slower, BF16, d = 128), but none wider than
    // the centres need: 2M x 128, split, k = 30: 64-wide 217 us, 128-wide 308, 256-wide
    // 369; k = 100: 314 (128-wide), 370; BF16, d = 64, k = 8: 152, 168, 222; k = 100: 186
    // (128-wide), 191
    const int N = k <= 64 ? 64 : k <= 128 ? 128 : TC_N;
    one[0] = TcPlanInst{x, ldx, n, d, centres, k, labels, 0, N, split};
    GK_TRY(tc_plan_build(ctx, &scr, one, P, st));
    return tc_plan_enqueue(ctx, *P, flag_rows, flag_m, n_flag, st);
}

// ---- candidates of the flagged rows ------------------------------------------
namespace {

// Slot s of the wave starting at unit u0: the flagged row's stored BF16 row
// (warp per slot, 16 bytes per lane) and its limit m + 2W: every centre that
// can be the exact argmin has a fast value of at most that (m: the smallest
// fast value the first pass saw, W the rigorous half-window of the mode).  A
// slot without a row, or whose limit is not finite, gets -inf: no candidate.
__global__ void __launch_bounds__(256) k_gather_flagged(const TcInst *__restrict__ inst, const TcXPrep *__restrict__ X,
                                                        const int64_t *__restrict__ row_off, FlagUnits F,
                                                        const float *__restrict__ mrow, int64_t u0, int64_t umax,
                                                        __nv_bfloat16 *__restrict__ xg, int kg,
                                                        float *__restrict__ lim) {
    const int lane = threadIdx.x & 31;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t nslots = TC_M * max((int64_t)0, min(umax, (int64_t)*F.n_units - u0));
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslots; s += nw) {
        const int64_t u = u0 + s / TC_M;
        const int r = (int)(s % TC_M), ii = F.unit_inst[u];
        float l = -INFINITY;
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (r < F.unit_cnt[u]) {
            const int64_t g = F.grows[F.unit_start[u] + r], i = g - row_off[ii];
            const TcXPrep &P = X[ii];
            const TcInst &I = inst[ii];
            const int W = P.split ? 2 * P.Kp : P.Kp;
            if (8 * lane < W) v = *reinterpret_cast<const uint4 *>(P.xb + i * W + 8 * lane);
            const float cmax = sqrtf(__uint_as_float(*I.cmax_bits)) * (1.f + 1e-5f);
            const float w2 = 2.f * (P.split ? window_bf16x3(I.xnorm[i], cmax, P.d) : window_bf16(I.xnorm[i], cmax, P.d));
            const float m = mrow[g], q = fmaf(w2, 1.f + 1e-6f, m) + fabsf(m) * 1.2e-7f;
            if (fabsf(q) < FLT_MAX) l = q;
        }
        if (8 * lane < kg) *reinterpret_cast<uint4 *>(xg + s * kg + 8 * lane) = v;
        if (lane == 0) lim[s] = l;
    }
}

// The exact argmin among a flagged row's candidates.  The direct distance D =
// sum (x - c)^2 in FP32 has none of the cancellation of |c|^2 - 2 x.c: with u =
// 2^-24, C = max |c| and D' its FP32 value (centres rounded to FP32,
// differences, FMA chains over the lanes and a shuffle tree),
//   |D' - D| <= ((d + 6) u D' + 2.001 u C sqrt(D') + 4.1 u^2 C^2)(1 + 10^-4)
// (|x - c32| is off by u|x - c32| + u|c| per coordinate, Cauchy-Schwarz over the
// coordinates, gamma_(d+4) for the sum), and the FP64 reference's own error
// is below d 2^-52 D; cand_err rounds all of it up by 5 %.  Where the smallest
// D' is apart from the second by both errors the label is decided; else (and
// without a candidate) the row goes on to `left`, for the FP32 scan and the
// FP64 reference.
__device__ __forceinline__ float cand_err(float D, float C, int d) {
    const float u = 5.9604645e-8f;
    return 1.05f * ((float)(d + 6) * u * D + 2.001f * u * C * sqrtf(D) + 4.1f * u * u * C * C) + 1e-37f;
}

// coordinates t .. t + 3, zeros past d
__device__ __forceinline__ float4 cand_load4(const float *__restrict__ p, int t, int d, bool vec) {
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (vec) {
        if (t < d) v = *reinterpret_cast<const float4 *>(p + t);
    } else {
        if (t < d) v.x = p[t];
        if (t + 1 < d) v.y = p[t + 1];
        if (t + 2 < d) v.z = p[t + 2];
        if (t + 3 < d) v.w = p[t + 3];
    }
    return v;
}
__device__ __forceinline__ bool cand_vec(const RInst &I) {
    return ((I.d & 3) == 0) && ((I.ldx & 3) == 0) && ((((uintptr_t)I.x) | ((uintptr_t)I.c32)) & 15) == 0;
}

// the set bits of the warp's 32 words (a word per lane) as a list; its length
__device__ __forceinline__ int cand_list(uint32_t m, uint16_t *list) {
    const int lane = threadIdx.x & 31, mine = __popc(m);
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += y;
    }
    __syncwarp();
    for (int at = inc - mine; m; m &= m - 1, at++) list[at] = (uint16_t)(32 * lane + __ffs((int)m) - 1);
    __syncwarp();
    return __shfl_sync(0xffffffffu, inc, 31);
}

// A row (in label order: 8 rows together) with more candidates than k / part goes
// to the FP32 scan of every centre.  Data far from the origin (|x| a hundred
// times the spread in BF16) make every centre a candidate, and a pair then costs
// 73 ps here (48 per centre of the union of 8 rows) against 9 ps in the scan, or
// 32 where that leaves the row to the FP64 reference: part = 6 and 4 lie between.
// Scan tiles are 64 centres wide, so up to 64 candidates stay.
// 90,000 x 128 in BF16, k = 2,000, all of them candidates: 1.9 ms, 13.1 by direct
// distances; 600,000 rows in label order 10.9 ms, 57.4 by direct distances.
__device__ __forceinline__ int cand_most(int64_t k, int part) { return (int)max((int64_t)64, k / part); }

// Rows in the order of their labels (decide_flags with an order): a warp takes 8
// neighbouring slots, whose candidates are nearly the same, and computes the
// distances of all 8 to the union (a real distance of a centre that is no
// candidate changes nothing).  A centre is read once for 8 rows: each eight-lane
// group holds two rows, lane l the coordinates 4 l .. 4 l + 3 of each 32, and all
// groups read the same 128-byte line.  Per (row, centre) pair that is about 6
// instructions with packed FP32 arithmetic; a warp per row, a candidate per
// group, took 43 and waited for L2.
__global__ void __launch_bounds__(256) k_decide_ordered(const RInst *__restrict__ R, FlagUnits F, int64_t u0,
                                                        int64_t umax, const uint32_t *__restrict__ masks, int kw,
                                                        int32_t *__restrict__ left,
                                                        unsigned long long *__restrict__ n_left) {
    __shared__ uint16_t s_list[8][1024];
    const int lane = threadIdx.x & 31, grp = lane >> 3, sub = lane & 7;
    uint16_t *list = s_list[threadIdx.x >> 5];
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t nsets = (TC_M / 8) * max((int64_t)0, min(umax, (int64_t)*F.n_units - u0));
    for (int64_t q8 = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; q8 < nsets; q8 += nw) {
        const int64_t u = u0 + q8 / (TC_M / 8), s = 8 * q8;  // s: slot in the wave
        const int r0 = (int)(q8 % (TC_M / 8)) * 8, cnt = F.unit_cnt[u];
        if (r0 >= cnt) continue;
        const RInst &I = R[F.unit_inst[u]];
        const int d = I.d;
        const bool vec = cand_vec(I);
        int64_t g[2];
        unsigned long long nx[2][8];  // -x in pairs
        bool row[2];
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const int r = r0 + grp + 4 * h;
            row[h] = r < cnt;
            g[h] = row[h] ? (int64_t)F.grows[F.unit_start[u] + r] : I.row_base;
#pragma unroll
            for (int e = 0; e < 4; e++) {
                const float4 v = cand_load4(I.x + (g[h] - I.row_base) * I.ldx, 32 * e + 4 * sub, d, vec);
                asm("mov.b64 %0, {%1, %2};" : "=l"(nx[h][2 * e]) : "f"(-v.x), "f"(-v.y));
                asm("mov.b64 %0, {%1, %2};" : "=l"(nx[h][2 * e + 1]) : "f"(-v.z), "f"(-v.w));
            }
        }
        const int nwords = (int)((I.k + 31) >> 5);
        int n_union = 0;
        for (int w = lane; w < nwords; w += 32) {
            uint32_t m = 0;
#pragma unroll
            for (int r = 0; r < 8; r++) m |= r0 + r < cnt ? masks[(s + r) * kw + w] : 0u;
            n_union += __popc(m);
        }
        n_union = __reduce_add_sync(0xffffffffu, n_union);
        if (n_union > cand_most(I.k, 4)) {
            const int rows = min(8, cnt - r0);
            unsigned long long at = 0;
            if (lane == 0) at = atomicAdd(n_left, (unsigned long long)rows);
            at = __shfl_sync(0xffffffffu, at, 0);
            if (lane < rows) left[at + lane] = F.grows[F.unit_start[u] + r0 + lane];
            continue;
        }
        float b1[2] = {FLT_MAX, FLT_MAX}, b2[2] = {FLT_MAX, FLT_MAX};
        int bj[2] = {0x7FFFFFFF, 0x7FFFFFFF}, total = 0;
        uint32_t own = 0;  // bit r: slot s + r has a candidate
        bool bad = false;
        for (int w0 = 0; w0 < nwords; w0 += 32) {
            uint32_t m = 0;
#pragma unroll
            for (int r = 0; r < 8; r++) {
                uint32_t w = w0 + lane < nwords && r0 + r < cnt ? masks[(s + r) * kw + w0 + lane] : 0u;
                // no index past the centres
                if (w0 + lane == nwords - 1 && (I.k & 31)) w &= (1u << (I.k & 31)) - 1u;
                if (__any_sync(0xffffffffu, w != 0)) own |= 1u << r;
                m |= w;
            }
            const int nc = cand_list(m, list);
            total += nc;
#pragma unroll 2
            for (int q = 0; q < nc; q++) {
                const int j = 32 * w0 + (int)list[q];
                const float *c = I.c32 + (int64_t)j * d;
                unsigned long long acc[2] = {0ull, 0ull};
#pragma unroll
                for (int e = 0; e < 4; e++) {
                    if (32 * e >= d) break;
                    const float4 cv = cand_load4(c, 32 * e + 4 * sub, d, vec);
                    unsigned long long c01, c23;
                    asm("mov.b64 %0, {%1, %2};" : "=l"(c01) : "f"(cv.x), "f"(cv.y));
                    asm("mov.b64 %0, {%1, %2};" : "=l"(c23) : "f"(cv.z), "f"(cv.w));
#pragma unroll
                    for (int h = 0; h < 2; h++) {
                        unsigned long long d01, d23;
                        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d01) : "l"(c01), "l"(nx[h][2 * e]));
                        asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d23) : "l"(c23), "l"(nx[h][2 * e + 1]));
                        asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(acc[h]) : "l"(d01));
                        asm("fma.rn.f32x2 %0, %1, %1, %0;" : "+l"(acc[h]) : "l"(d23));
                    }
                }
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    float D = __uint_as_float((uint32_t)acc[h]) + __uint_as_float((uint32_t)(acc[h] >> 32));
#pragma unroll
                    for (int o = 1; o < 8; o <<= 1) D += __shfl_xor_sync(0xffffffffu, D, o);
                    bad = bad || !(D < FLT_MAX);
                    const bool less = D < b1[h];
                    b2[h] = fminf(b2[h], less ? b1[h] : D);
                    b1[h] = less ? D : b1[h];
                    bj[h] = less ? j : bj[h];
                }
            }
        }
        if (sub == 0) {
            const float C = __uint_as_float(*I.cmax_bits);
#pragma unroll
            for (int h = 0; h < 2; h++) {
                if (!row[h]) continue;
                const bool sure = !bad && ((own >> (grp + 4 * h)) & 1u) &&
                                  (total == 1 || (b2[h] - b1[h]) * (1.f - 1e-6f) > cand_err(b1[h], C, d) + cand_err(b2[h], C, d));
                if (sure) I.labels[g[h] - I.row_base] = bj[h];
                else left[atomicAdd(n_left, 1ull)] = (int32_t)g[h];
            }
        }
    }
}

// Rows in any order: a warp per slot, its eight-lane groups take a candidate
// each, two in flight.
__global__ void __launch_bounds__(256) k_decide_candidates(const RInst *__restrict__ R, FlagUnits F, int64_t u0,
                                                           int64_t umax, const uint32_t *__restrict__ masks, int kw,
                                                           int32_t *__restrict__ left,
                                                           unsigned long long *__restrict__ n_left) {
    __shared__ uint16_t s_list[8][1024];
    const int lane = threadIdx.x & 31, grp = lane >> 3, sub = lane & 7;
    uint16_t *list = s_list[threadIdx.x >> 5];
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t nslots = TC_M * max((int64_t)0, min(umax, (int64_t)*F.n_units - u0));
    for (int64_t s = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; s < nslots; s += nw) {
        const int64_t u = u0 + s / TC_M;
        const int r = (int)(s % TC_M);
        if (r >= F.unit_cnt[u]) continue;
        const RInst &I = R[F.unit_inst[u]];
        const int64_t g = F.grows[F.unit_start[u] + r], row = g - I.row_base;
        const int d = I.d;
        const bool vec = cand_vec(I);
        float4 xv[4];
#pragma unroll
        for (int q = 0; q < 4; q++) xv[q] = cand_load4(I.x + row * I.ldx, 32 * q + 4 * sub, d, vec);
        const uint32_t *mk = masks + s * kw;
        const int nwords = (int)((I.k + 31) >> 5);
        int n_cand = 0;
        for (int w = lane; w < nwords; w += 32) n_cand += __popc(mk[w]);
        n_cand = __reduce_add_sync(0xffffffffu, n_cand);
        if (n_cand > cand_most(I.k, 6)) {
            if (lane == 0) left[atomicAdd(n_left, 1ull)] = (int32_t)g;
            continue;
        }
        float b1 = FLT_MAX, b2 = FLT_MAX;  // this group's smallest and second D'
        int bj = 0x7FFFFFFF, total = 0;
        bool bad = false;
        for (int w0 = 0; w0 < nwords; w0 += 32) {
            uint32_t m = w0 + lane < nwords ? mk[w0 + lane] : 0u;
            if (w0 + lane == nwords - 1 && (I.k & 31)) m &= (1u << (I.k & 31)) - 1u;  // no index past the centres
            const int cnt = cand_list(m, list);
            total += cnt;
            for (int q0 = 0; q0 < cnt; q0 += 8) {  // two candidates per group in flight
                float D[2];
                int j[2];
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    const int q = q0 + 4 * h + grp;
                    j[h] = q < cnt ? 32 * w0 + (int)list[q] : -1;
                    const float *c = I.c32 + (int64_t)max(j[h], 0) * d;
                    D[h] = 0.f;
#pragma unroll
                    for (int e = 0; e < 4; e++) {
                        if (32 * e >= d) break;
                        const float4 cv = cand_load4(c, 32 * e + 4 * sub, d, vec);
                        const float e0 = xv[e].x - cv.x, e1 = xv[e].y - cv.y;
                        const float e2 = xv[e].z - cv.z, e3 = xv[e].w - cv.w;
                        D[h] = fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, fmaf(e0, e0, D[h]))));
                    }
                }
#pragma unroll
                for (int o = 1; o < 8; o <<= 1) {
                    D[0] += __shfl_xor_sync(0xffffffffu, D[0], o);
                    D[1] += __shfl_xor_sync(0xffffffffu, D[1], o);
                }
#pragma unroll
                for (int h = 0; h < 2; h++) {
                    if (j[h] < 0) continue;
                    bad = bad || !(D[h] < FLT_MAX);
                    if (D[h] < b1) {
                        b2 = b1;
                        b1 = D[h];
                        bj = j[h];
                    } else {
                        b2 = fminf(b2, D[h]);
                    }
                }
            }
        }
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) {  // the four groups
            const float o1 = __shfl_xor_sync(0xffffffffu, b1, o), o2 = __shfl_xor_sync(0xffffffffu, b2, o);
            const int oj = __shfl_xor_sync(0xffffffffu, bj, o);
            b2 = fminf(fminf(b2, o2), fmaxf(b1, o1));
            if (o1 < b1) bj = oj;
            b1 = fminf(b1, o1);
        }
        bad = __any_sync(0xffffffffu, bad);
        if (lane == 0) {
            const float C = __uint_as_float(*I.cmax_bits);
            const bool sure = !bad && (total == 1 || (total > 1 && (b2 - b1) * (1.f - 1e-6f) >
                                                                       cand_err(b1, C, d) + cand_err(b2, C, d)));
            if (sure) I.labels[row] = bj;
            else left[atomicAdd(n_left, 1ull)] = (int32_t)g;
        }
    }
}

}  // namespace

// The plan's part of the exact decision: per wave of flagged units (grouped by
// decide_flags: F, every row's smallest value in mrow), gather the rows, find
// their candidates with a second tcgen05 pass over them, and decide among the
// candidates; what stays undecided is appended to left / n_left.  max_rows
// bounds the flagged rows; ordered: they are in the order of their labels.  No
// allocation and no host synchronisation (the buffers are the plan's,
// tc_emit_alloc).
geek_status tc_decide_candidates(geek_ctx *ctx, const TcPlan &P, const RInst *R, const FlagUnits &F, const float *mrow,
                                 int64_t max_rows, bool ordered, int32_t *left, unsigned long long *n_left,
                                 cudaStream_t st) {
    int64_t units = ceil_div(std::min(max_rows, P.N_total), TC_M) + P.count;
    bool mode[2] = {false, false};
    for (const TcPlanInst &I : P.desc)
        if (I.n > 0 && I.k > 0) mode[I.split ? 1 : 0] = true;
    EvTimer tk(ctx, "kernel.assign_candidates", st);
    for (int64_t u0 = 0; u0 < units; u0 += P.emit_units) {
        GK_COUNT();
        k_gather_flagged<<<ctx->num_sms * 8, 256, 0, st>>>(P.inst, P.xprep, P.row_off, F, mrow, u0, P.emit_units,
                                                           P.xg, P.kg, P.emit_lim);
        TcArgs A{};
        A.inst = P.inst;
        A.nunits = P.emit_units;
        A.err = P.err;
        A.e = TcEmit{P.tmG, P.emit_lim, P.emit_masks, P.kw, F.unit_inst, F.n_units, u0};
        for (int sp = 0; sp < 2; sp++) {
            if (!mode[sp]) continue;
            const Rings r = ring_lg(P, nullptr, sp);
            A.lg_ns = r.ns;
            A.lg_nx = r.nx;
            A.lg_na = r.na;
            GK_COUNT();
            const int grid = (int)std::min<int64_t>(P.emit_units, ctx->num_sms);
            if (sp) k_assign_tc<true, true><<<grid, TC_THREADS, tc_smem(), st>>>(A);
            else k_assign_tc<false, true><<<grid, TC_THREADS, tc_smem(), st>>>(A);
        }
        GK_COUNT();
        (ordered ? k_decide_ordered : k_decide_candidates)<<<ctx->num_sms * 8, 256, 0, st>>>(
            R, F, u0, P.emit_units, P.emit_masks, P.kw, left, n_left);
        GK_LAUNCH(ctx);
    }
    return GEEK_OK;
}

// Buffers of tc_decide_candidates for at most max_rows flagged rows: a wave
// holds as many units as fit EMIT_BYTES (gathered rows and masks), at least one,
// and as many as the device has room for: with half the units there are twice
// the waves and the same labels, so a request that fails is halved (down to
// EMIT_WAVES waves for a batch, whose graph holds a few launches per wave).
geek_status tc_emit_alloc(geek_ctx *ctx, Scratch *scr, TcPlan *P, int64_t max_rows, cudaStream_t st) {
    constexpr int64_t EMIT_BYTES = 1ll << 30, EMIT_WAVES = 4096;
    int kg = 64;
    int64_t kw = 8;
    for (const TcPlanInst &I : P->desc) {
        const int Kp = I.d <= 64 ? 64 : 128;
        kg = std::max(kg, (I.split || P->allow_split) ? 2 * Kp : Kp);
        kw = std::max(kw, ceil_div(I.k, TC_N) * (TC_N / 32));
    }
    // one block: the tensor map, then per unit rows, masks and limits (all
    // multiples of 256 bytes)
    const int64_t row_bytes = TC_M * 2 * (int64_t)kg, mask_bytes = TC_M * 4 * kw, lim_bytes = TC_M * 4;
    const int64_t all = ceil_div(std::min(max_rows, P->N_total), TC_M) + P->count;
    int64_t units = std::min(all, std::max<int64_t>(EMIT_BYTES / (row_bytes + mask_bytes + lim_bytes), 1));
    const int64_t least = scr ? 1 : std::min(units, ceil_div(all, EMIT_WAVES));
    char *block = nullptr;
    const std::string msg = ctx->last_error;
    for (;;) {
        const geek_status rc = plan_alloc(ctx, scr, P->owned, &block,
                                          (size_t)(256 + units * (row_bytes + mask_bytes + lim_bytes)));
        if (rc == GEEK_OK) break;
        if (rc != GEEK_ERR_NOMEM || units <= least) return rc;
        units = std::max(least, units / 2);
        ctx->last_error = msg;  // nothing has failed yet
    }
    P->kg = kg;
    P->kw = (int)kw;
    P->emit_units = units;
    P->tmG = (CUtensorMap *)block;
    P->xg = (__nv_bfloat16 *)(block + 256);
    P->emit_masks = (uint32_t *)(block + 256 + units * row_bytes);
    P->emit_lim = (float *)(block + 256 + units * (row_bytes + mask_bytes));
    CUtensorMap tm;
    GK_TRY(encode_bf16_2d(ctx, &tm, P->xg, kg, (uint64_t)(units * TC_M), TC_KB, TC_M));
    GK_CUDA(ctx, cudaMemcpyAsync(P->tmG, &tm, sizeof tm, cudaMemcpyHostToDevice, st));
    return GEEK_OK;
}
