// Central vectors and one-pass data assignment (Sect. 3.3, Eq. 1).
//
// Dense assignment evaluates d'_j = |c_j|^2 - 2 x.c_j (the row-constant
// |x|^2 dropped) for every centre in a fast precision, keeps the best and
// second-best value per object, and decides the argmin in FP64 only for
// objects whose gap is within the rigorous error window.  The FP64 decision
// reproduces the reference distance exactly: sum_t ((double)x_t - c_t)^2 in t
// order, each operation rounded to nearest, no fused multiply-add; ties go
// to the smallest centre index.
#include <cfloat>
#include <cstddef>
#include <type_traits>

#include "internal.cuh"
#include "tc_ptx.cuh"

namespace {

constexpr int AS_TR = 128;   // rows per block
constexpr int AS_TC = 64;    // centres per tile
constexpr int AS_KC = 32;    // d-chunk of the centre tile
constexpr int AS_RPT = 8;    // rows per thread
constexpr int AS_CPT = 4;    // centres per thread
constexpr int AS_MAXD = 256; // X tile resident in shared memory

struct Best {
    float b1, b2;
    int i1;
};

__device__ __forceinline__ void best_push(Best &B, float v, int j) {
    if (v < B.b1) {
        B.b2 = B.b1;
        B.b1 = v;
        B.i1 = j;
    } else {
        B.b2 = fminf(B.b2, v);
    }
}

__device__ __forceinline__ Best best_merge(Best a, Best b) {
    Best r;
    const bool take_b = b.b1 < a.b1 || (b.b1 == a.b1 && b.i1 < a.i1);
    r.b1 = take_b ? b.b1 : a.b1;
    r.i1 = take_b ? b.i1 : a.i1;
    r.b2 = fminf(fminf(a.b2, b.b2), take_b ? a.b1 : b.b1);
    return r;
}

// FP32 SIMT assignment: block = 128 rows, all centres streamed in tiles of
// 64; 256 threads = 16 row groups x 16 centre groups, a thread the rows rg +
// 16 r (r < 8) and the centres cg + 16 c (c < 4) of a tile.
// The FP32 pipe bounds it, so everything else is kept off the issue slots:
// packed FMAs (fma.rn.f32x2, two products per instruction: the even and the
// odd coordinates of a product sum apart and are added at the end, within the
// window, which holds for any order of the d terms), operands as 16-byte
// shared-memory loads of four consecutive coordinates, 12 loads per 64 packed
// FMAs.  Rows are stored coordinate-contiguous with their 16-byte pieces
// XOR-swizzled by the row, so the 2 rows and the 16 centres a warp reads at
// once fall into different banks; the centre chunks (64 x 32) arrive by
// cp.async two chunks ahead in a ring of three (fp32_narrow: in chunks of 16, one ahead).
// n = 1,000,003, d = 96, k = 2,000: the call takes 11.9 ms, against 14.6 ms with
// scalar FMAs on transposed tiles, whose fills were 32-way bank conflicts.
// GATHER = false: blocks walk the row tiles of the one data set A.
// GATHER = true: blocks walk units of up to 128 flagged rows of one instance
// (unit u: instance unit_inst[u], global rows grows[unit_start[u] ..
// + unit_cnt[u]]); the instance's data replace A's, uncertain rows are
// appended (as global rows) to A.flag_rows.
struct FArgs {
    const float *x;
    int64_t ldx, n;
    int d;
    const float *c32, *cn;
    int64_t k;
    const unsigned *cmax_bits;
    int32_t *labels;
    int32_t *flag_rows;
    float *flag_m;  // may be null: the row's smallest fast value, beside flag_rows
    unsigned long long *n_flag;
    int64_t ntiles;
};
struct GatherUnits {
    const RInst *R;
    FlagUnits f;
};

// c += a b, two FP32 values each
__device__ __forceinline__ void ffma2(unsigned long long &c, unsigned long long a, unsigned long long b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(a), "l"(b));
}

// The centre ring: KC coordinates of the 64 centres per stage, ST stages.  Three
// of 32 where two blocks fit an SM (d <= 160), or where no form lets them (d >
// 208); between, with more than one block per SM, two of 16, with which two fit:
// one alone has nothing to do while its rows arrive (1M x 200, k = 50: 1.40 ms,
// 1.71 with one block; k = 1,000, 300,000 rows: 4.0 ms, 4.7).  With one block per
// SM anyway the longer ring is the faster one (2,000 x 200, k = 3,000: 0.91, 1.00).
static bool fp32_narrow(const geek_ctx *ctx, int64_t n, int d) {
    return d > 160 && d <= 208 && n > (int64_t)ctx->num_sms * AS_TR;
}
// shared memory of k_assign_fp32: the row tile, coordinates padded to whole
// chunks, and the centre ring
static size_t fp32_smem(int d, bool narrow) {
    const int kc = narrow ? 16 : 32, st = narrow ? 2 : 3;
    return ((size_t)AS_TR * ((d + kc - 1) / kc * kc) + st * AS_TC * kc) * sizeof(float);
}

template <bool GATHER, int KC, int ST>
__global__ void __launch_bounds__(256, 2) k_assign_fp32(FArgs A, GatherUnits U) {
    constexpr int CST = AS_TC * KC, PC = KC / 4;  // floats per stage, 16-byte pieces per chunk and centre
    extern __shared__ __align__(16) float sm[];
    __shared__ int64_t s_rows[AS_TR];
    const int t = threadIdx.x, cg = t & 15, rg = t >> 4;
    const int64_t nunits = GATHER ? (int64_t)*U.f.n_units : A.ntiles;
    for (int64_t u = blockIdx.x; u < nunits; u += gridDim.x) {
        int64_t row0 = u * AS_TR;
        int nrows = (int)min((int64_t)AS_TR, A.n - row0);
        int64_t rbase = 0;
        if (GATHER) {
            const RInst &I = U.R[U.f.unit_inst[u]];
            A.x = I.x;
            A.ldx = I.ldx;
            A.d = I.d;
            A.c32 = I.c32;
            A.cn = I.cn;
            A.k = I.k;
            A.cmax_bits = I.cmax_bits;
            A.labels = I.labels;
            rbase = I.row_base;
            nrows = U.f.unit_cnt[u];
            __syncthreads();  // s_rows of the previous unit fully used
            if (t < nrows) s_rows[t] = (int64_t)U.f.grows[U.f.unit_start[u] + t] - rbase;
            __syncthreads();
        }
        const int d = A.d;
        const int64_t k = A.k;
        const int nch = (d + KC - 1) / KC;         // chunks of KC coordinates
        const int dp = nch * KC, dp16 = 16 * dp;
        float *xs = sm;                            // [AS_TR][dp], pieces swizzled
        float *cs = sm + (size_t)AS_TR * dp;       // [ST][AS_TC][KC], pieces swizzled
        // rows of an odd number of 64-byte halves fall into different banks by themselves
        const int xm = (dp & 16) ? 0 : 7;
        const bool xvec = ((A.ldx & 3) == 0) && ((d & 3) == 0) && (((uintptr_t)A.x & 15) == 0);
        const bool cvec = ((d & 3) == 0) && (((uintptr_t)A.c32 & 15) == 0);
        const int ntile = (int)((k + AS_TC - 1) / AS_TC);
        // 16-byte piece p of row r at position p ^ (r & 7) within each group of
        // eight pieces (of four in a 16-coordinate centre chunk, where two centres
        // span the banks: p ^ (c / 2 & 3)); zeros outside the data.  Rows without
        // 16-byte alignment arrive as asynchronously, by 4-byte copies (1M x 150, k
        // = 50: 1.14 ms, 1.29 with loads and stores).
        auto put = [&](float *dst, const float *src, int nv, bool vec) {
            if (vec) {
                asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(
                                 (uint32_t)__cvta_generic_to_shared(dst)),
                             "l"(nv > 0 ? src : A.c32), "r"(nv > 0 ? 16 : 0)
                             : "memory");
            } else {
#pragma unroll
                for (int q = 0; q < 4; q++)
                    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(
                                     (uint32_t)__cvta_generic_to_shared(dst + q)),
                                 "l"(q < nv ? src + q : A.c32), "r"(q < nv ? 4 : 0)
                                 : "memory");
            }
        };
        auto centre_piece = [](int c, int p) { return KC == 32 ? p ^ (c & 7) : p ^ ((c >> 1) & 3); };
        // the next chunk (tile f_t, chunk f_c) into ring slot f_s; counters instead
        // of divisions of a chunk number, which cost as much as the products
        int f_t = 0, f_c = 0, f_s = 0;
        auto stage = [&]() {
            if (f_t < ntile) {
                const int k0 = f_c * KC;
                float *buf = cs + f_s * CST;
#pragma unroll
                for (int u = 0; u < CST / 4 / 256; u++) {
                    const int e = t + 256 * u, c = e / PC, p = e % PC;
                    const int64_t j = (int64_t)f_t * AS_TC + c;
                    put(buf + c * KC + 4 * centre_piece(c, p), A.c32 + j * d + k0 + 4 * p,
                        j < k ? min(4, d - k0 - 4 * p) : 0, cvec);
                }
                if (++f_c == nch) f_c = 0, f_t++;
                if (++f_s == ST) f_s = 0;
            }
            asm volatile("cp.async.commit_group;" ::: "memory");
        };
        __syncthreads();  // the previous unit's tile fully used
        for (int e = t; e < AS_TR * (dp >> 2); e += 256) {
            const int r = e / (dp >> 2), p = e % (dp >> 2);
            const int64_t row = r < nrows ? (GATHER ? s_rows[r] : row0 + r) : 0;
            put(xs + r * dp + 4 * (p ^ (r & xm)), A.x + row * A.ldx + 4 * p, r < nrows ? min(4, d - 4 * p) : 0, xvec);
        }
#pragma unroll
        for (int u = 0; u < ST - 1; u++) stage();
        Best B[AS_RPT];
#pragma unroll
        for (int r = 0; r < AS_RPT; r++) B[r] = Best{FLT_MAX, FLT_MAX, 0x7FFFFFFF};
        unsigned long long acc[AS_RPT][AS_CPT];
        int ch = 0, slot = 0;
        for (int tile = 0; tile < ntile;) {
            asm volatile("cp.async.wait_group %0;" ::"n"(ST - 2) : "memory");
            __syncthreads();  // this chunk has landed; everyone is done with the last one's slot
            stage();
            if (ch == 0) {
#pragma unroll
                for (int r = 0; r < AS_RPT; r++)
#pragma unroll
                    for (int c = 0; c < AS_CPT; c++) acc[r][c] = 0ull;
            }
            const float *buf = cs + slot * CST + cg * KC, *xb = xs + rg * dp;
            if (++slot == ST) slot = 0;
            const int np = min(KC, d - ch * KC + 3) >> 2;  // pieces holding data
#pragma unroll 1
            for (int p = 0; p < np; p++) {
                ulonglong2 cv[AS_CPT];
#pragma unroll
                for (int c = 0; c < AS_CPT; c++)  // centre_piece(cg + 16 c, p) is centre_piece(cg, p)
                    cv[c] = *reinterpret_cast<const ulonglong2 *>(buf + 16 * c * KC + 4 * centre_piece(cg, p));
#pragma unroll
                for (int r = 0; r < AS_RPT; r++) {
                    const ulonglong2 xv = *reinterpret_cast<const ulonglong2 *>(xb + r * dp16 + 4 * ((ch * PC + p) ^ (rg & xm)));
#pragma unroll
                    for (int c = 0; c < AS_CPT; c++) {
                        ffma2(acc[r][c], xv.x, cv[c].x);
                        ffma2(acc[r][c], xv.y, cv[c].y);
                    }
                }
            }
            if (++ch == nch) {
                ch = 0;
#pragma unroll
                for (int c = 0; c < AS_CPT; c++) {
                    const int j = tile * AS_TC + cg + 16 * c;
                    if (j >= k) continue;
                    const float cnj = A.cn[j];
#pragma unroll
                    for (int r = 0; r < AS_RPT; r++) {
                        const float dot = __uint_as_float((uint32_t)acc[r][c]) + __uint_as_float((uint32_t)(acc[r][c] >> 32));
                        best_push(B[r], fmaf(-2.f, dot, cnj), j);
                    }
                }
                tile++;
            }
        }
        asm volatile("cp.async.wait_group 0;" ::: "memory");
        // merge the 16 centre groups of each row group (lanes of one half-warp)
#pragma unroll
        for (int r = 0; r < AS_RPT; r++) {
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) {
                Best o_;
                o_.b1 = __shfl_xor_sync(0xffffffffu, B[r].b1, o);
                o_.b2 = __shfl_xor_sync(0xffffffffu, B[r].b2, o);
                o_.i1 = __shfl_xor_sync(0xffffffffu, B[r].i1, o);
                B[r] = best_merge(B[r], o_);
            }
        }
        const float cmax = __uint_as_float(*A.cmax_bits);
        // |x|^2 of the row group's rows, the coordinates over its 16 lanes
        float xs2[AS_RPT];
#pragma unroll
        for (int r = 0; r < AS_RPT; r++) {
            xs2[r] = 0.f;
            for (int p = cg; p < (dp >> 2); p += 16) {
                const float4 v = *reinterpret_cast<const float4 *>(xs + (rg + 16 * r) * dp + 4 * (p ^ (rg & xm)));
                xs2[r] = fmaf(v.x, v.x, fmaf(v.y, v.y, fmaf(v.z, v.z, fmaf(v.w, v.w, xs2[r]))));
            }
#pragma unroll
            for (int o = 1; o < 16; o <<= 1) xs2[r] += __shfl_xor_sync(0xffffffffu, xs2[r], o);
        }
        if (cg == 0) {
#pragma unroll
            for (int r = 0; r < AS_RPT; r++) {
                const int rr = rg + 16 * r;
                if (rr >= nrows) continue;
                const int64_t row = GATHER ? s_rows[rr] : row0 + rr;
                const float xn = sqrtf(xs2[r]) * (1.f + 1.0e-3f);
                const float W = 2.f * window_fp32(xn, cmax, d);
                // no finite value (non-finite input): undecided here, FP64 decides
                const bool valid = B[r].i1 != 0x7FFFFFFF;
                A.labels[row] = valid ? B[r].i1 : -1;
                const bool sure = valid && (k == 1 || (B[r].b2 - B[r].b1 > W * (1.f + 1e-6f)));
                if (!sure) {
                    const unsigned long long q = atomicAdd(A.n_flag, 1ull);
                    A.flag_rows[q] = (int32_t)(rbase + row);
                    if (A.flag_m) A.flag_m[q] = valid ? B[r].b1 : __int_as_float(0x7fc00000);
                }
            }
        }
    }
}

// The tiled FP64 decision of the rows the FP32 refine leaves uncertain: the
// centres streamed through shared memory in tiles, the FP32 fast value of
// every (row, centre) pair in registers.  A pair whose fast value lies within
// the row's window lim = m + 2W (m: the row's smallest fast value, from the
// refine pass, in mrow[global row]) gets the FP64 reference distance, read
// from the row in shared memory; the row's label is the smallest reference
// distance, ties to the smaller index (-1 when no value is finite).
//
// The FP64 distances are a chain of d dependent adds each, and the FP64 pipe
// issues one warp-wide operation about every 19 cycles per SM: computed by
// the thread that found the pair, one active lane would pay for a whole
// warp.  So the tile's pairs go to a shared-memory queue and the block takes
// them a lane each (in rounds of at most DQ_CAP pairs); each row's best is
// kept in shared memory as the smallest D (an atomic minimum on its bits: D
// >= 0, so the bit order is the value order), then the smallest index among
// the pairs that reach it.
constexpr int DQ_CAP = 2048;
constexpr size_t DQ_BYTES = (size_t)DQ_CAP * (sizeof(double) + sizeof(uint16_t));

// exact FP32 -> FP64 widening in integer operations (normal, subnormal, zero,
// infinity; a NaN stays a NaN): keeps the conversion off the FP64 pipe
__device__ __forceinline__ double widen_f32(float v) {
    const uint32_t b = __float_as_uint(v);
    const uint32_t sg = b & 0x80000000u, e = (b >> 23) & 0xFFu, m = b & 0x7FFFFFu;
    // subnormal: m = 1.f x 2^(p - 23) with p the top set bit, value m 2^-149
    const int sh = __clz((int)m) - 8;  // brings the top bit of m to bit 23
    const uint32_t ms = (m << (sh & 31)) & 0x7FFFFFu;
    const uint32_t es = (uint32_t)(1023 - 126 - sh);
    uint32_t hi, lo;
    if (e == 0u) {
        hi = m == 0u ? sg : (sg | (es << 20) | (ms >> 3));
        lo = m == 0u ? 0u : (ms << 29);
    } else {
        const uint32_t ed = e == 0xFFu ? 0x7FFu : e + 896u;
        hi = sg | (ed << 20) | (m >> 3);
        lo = m << 29;
    }
    return __hiloint2double((int)hi, (int)lo);
}

__device__ __forceinline__ double ref_dist_strided(const float *x, int stride, const double *__restrict__ c, int d) {
    double D = 0.0;
    for (int t = 0; t < d; t++) {
        const double e = __dsub_rn(widen_f32(x[t * stride]), c[t]);
        D = __dadd_rn(D, __dmul_rn(e, e));
    }
    return D;
}

__global__ void __launch_bounds__(256) k_assign_decide64(GatherUnits U, const float *__restrict__ mrow) {
    extern __shared__ float sm[];
    __shared__ float cns[AS_TC];
    __shared__ int64_t s_rows[AS_TR];
    __shared__ unsigned long long sbD[AS_TR], prevD[AS_TR];
    __shared__ int sbJ[AS_TR], tJ[AS_TR];
    __shared__ int s_qn;
    constexpr unsigned long long DINF = 0x7FF0000000000000ull;  // above every finite D
    const int t = threadIdx.x, cg = t & 15, rg = t >> 4;
    const int64_t nunits = (int64_t)*U.f.n_units;
    for (int64_t u = blockIdx.x; u < nunits; u += gridDim.x) {
        const RInst &I = U.R[U.f.unit_inst[u]];
        const int d = I.d;
        const int64_t k = I.k;
        const int64_t rbase = I.row_base;
        const int nrows = U.f.unit_cnt[u];
        __syncthreads();  // s_rows and xs of the previous unit fully used
        if (t < nrows) s_rows[t] = (int64_t)U.f.grows[U.f.unit_start[u] + t] - rbase;
        if (t < AS_TR) {
            sbD[t] = DINF;
            prevD[t] = DINF;
            sbJ[t] = 0x7FFFFFFF;
            tJ[t] = 0x7FFFFFFF;
        }
        if (t == 0) s_qn = 0;
        __syncthreads();
        float *xs = sm;                      // [d][AS_TR]
        float *cs = sm + (size_t)d * AS_TR;  // [AS_KC][AS_TC]
        double *qd = reinterpret_cast<double *>(cs + AS_KC * AS_TC);  // [DQ_CAP]
        uint16_t *qi = reinterpret_cast<uint16_t *>(qd + DQ_CAP);     // [DQ_CAP]: row * AS_TC + column
        for (int e = t; e < AS_TR * d; e += 256) {
            const int r = e / d, kk = e % d;
            xs[kk * AS_TR + r] = r < nrows ? I.x[s_rows[r] * I.ldx + kk] : 0.f;
        }
        __syncthreads();
        const float cmax = __uint_as_float(*I.cmax_bits);
        float lim[AS_RPT];
#pragma unroll
        for (int r = 0; r < AS_RPT; r++) {
            const int rr = rg * AS_RPT + r;
            float xs2 = 0.f;
            for (int kk = 0; kk < d; kk++) xs2 = fmaf(xs[kk * AS_TR + rr], xs[kk * AS_TR + rr], xs2);
            const float xn = sqrtf(xs2) * (1.f + 1.0e-3f);
            const float m = rr < nrows ? mrow[rbase + s_rows[rr]] : __int_as_float(0x7fc00000);
            lim[r] = m + 2.f * window_fp32(xn, cmax, d) * (1.f + 1e-6f);
        }
        for (int64_t j0 = 0; j0 < k; j0 += AS_TC) {
            float acc[AS_RPT][AS_CPT];
#pragma unroll
            for (int r = 0; r < AS_RPT; r++)
#pragma unroll
                for (int c = 0; c < AS_CPT; c++) acc[r][c] = 0.f;
            for (int k0 = 0; k0 < d; k0 += AS_KC) {
                __syncthreads();
                for (int e = t; e < AS_TC * AS_KC; e += 256) {
                    const int c = e / AS_KC, kk = e % AS_KC;
                    const int64_t j = j0 + c;
                    cs[kk * AS_TC + c] = (j < k && k0 + kk < d) ? I.c32[j * d + k0 + kk] : 0.f;
                }
                if (k0 == 0 && t < AS_TC) cns[t] = j0 + t < k ? I.cn[j0 + t] : FLT_MAX;
                __syncthreads();
                const int kmax = min(AS_KC, d - k0);
                for (int kk = 0; kk < kmax; kk++) {
                    const float4 x0 = *reinterpret_cast<const float4 *>(&xs[(k0 + kk) * AS_TR + rg * AS_RPT]);
                    const float4 x1 = *reinterpret_cast<const float4 *>(&xs[(k0 + kk) * AS_TR + rg * AS_RPT + 4]);
                    const float4 cv = *reinterpret_cast<const float4 *>(&cs[kk * AS_TC + cg * AS_CPT]);
                    const float xv[8] = {x0.x, x0.y, x0.z, x0.w, x1.x, x1.y, x1.z, x1.w};
                    const float cc[4] = {cv.x, cv.y, cv.z, cv.w};
#pragma unroll
                    for (int r = 0; r < AS_RPT; r++)
#pragma unroll
                        for (int c = 0; c < AS_CPT; c++) acc[r][c] = fmaf(xv[r], cc[c], acc[r][c]);
                }
            }
            // this thread's pairs inside the window: bit r * AS_CPT + c
            uint32_t pend = 0;
#pragma unroll
            for (int c = 0; c < AS_CPT; c++) {
                const int64_t j = j0 + cg * AS_CPT + c;
                const float cnj = cns[cg * AS_CPT + c];
#pragma unroll
                for (int r = 0; r < AS_RPT; r++) {
                    const int rr = rg * AS_RPT + r;
                    if (j < k && rr < nrows && fmaf(-2.f, acc[r][c], cnj) <= lim[r]) pend |= 1u << (r * AS_CPT + c);
                }
            }
            if (!__syncthreads_or(pend != 0)) continue;
            for (;;) {
                // queue what fits; the rest waits for the next round
                const int np = __popc(pend);
                int pos = np ? atomicAdd(&s_qn, np) : 0;
                uint32_t rest = 0;
                for (uint32_t m = pend; m; m &= m - 1) {
                    const int bt = __ffs((int)m) - 1;
                    if (pos < DQ_CAP)
                        qi[pos] = (uint16_t)((rg * AS_RPT + bt / AS_CPT) * AS_TC + cg * AS_CPT + bt % AS_CPT);
                    else
                        rest |= 1u << bt;
                    pos++;
                }
                pend = rest;
                __syncthreads();
                const int nq = min(s_qn, DQ_CAP);
                for (int e = t; e < nq; e += 256) {
                    const int ee = qi[e];
                    const int rr = ee / AS_TC;
                    const double D = ref_dist_strided(xs + rr, AS_TR, I.c64 + (j0 + ee % AS_TC) * d, d);
                    qd[e] = D;
                    atomicMin(&sbD[rr], (unsigned long long)__double_as_longlong(D));
                }
                __syncthreads();
                for (int e = t; e < nq; e += 256) {
                    const int ee = qi[e];
                    const int rr = ee / AS_TC;
                    if ((unsigned long long)__double_as_longlong(qd[e]) == sbD[rr])
                        atomicMin(&tJ[rr], (int)(j0 + ee % AS_TC));
                }
                __syncthreads();
                if (t < AS_TR) {
                    if (tJ[t] != 0x7FFFFFFF) {
                        // a new smallest D: its smallest index; the same D again: the smaller index
                        sbJ[t] = sbD[t] < prevD[t] ? tJ[t] : min(sbJ[t], tJ[t]);
                        tJ[t] = 0x7FFFFFFF;
                    }
                    prevD[t] = sbD[t];
                }
                if (t == 0) s_qn = 0;
                if (!__syncthreads_or(pend != 0)) break;
            }
        }
        if (t < nrows) I.labels[s_rows[t]] = sbJ[t] == 0x7FFFFFFF ? -1 : sbJ[t];
    }
}

__global__ void k_scatter_m(const int32_t *__restrict__ rows, const float *__restrict__ m,
                            const unsigned long long *__restrict__ n, float *__restrict__ mrow) {
    const int64_t nf = (int64_t)*n;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nf; q += (int64_t)gridDim.x * blockDim.x)
        mrow[rows[q]] = m[q];
}

// ---- grouping a flag list by instance (device-side, graph friendly) --------
// A warp adds once per instance among its 32 rows (neighbours in the list nearly
// always share theirs): 3.2M rows of 16 instances take 1.6 ms per kernel with an
// atomic per row, all of them on 16 words, and 65 us with one per warp.
__device__ __forceinline__ int flag_inst(const int32_t *__restrict__ flags, int64_t q, int64_t nf,
                                         const int64_t *__restrict__ row_off, int count, int32_t &r) {
    r = q < nf ? flags[q] : 0;
    return q < nf ? find_inst(row_off, count, r) : -1;
}
__global__ void k_flag_count(const int32_t *__restrict__ flags, const unsigned long long *__restrict__ n_flag,
                             const int64_t *__restrict__ row_off, int count, int *__restrict__ cnt) {
    const int64_t nf = (int64_t)*n_flag;
    const int lane = threadIdx.x & 31;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q - lane < nf;
         q += (int64_t)gridDim.x * blockDim.x) {
        int32_t r;
        const int i = flag_inst(flags, q, nf, row_off, count, r);
        const uint32_t peers = __match_any_sync(0xffffffffu, i);
        if (i >= 0 && lane == __ffs(peers) - 1) atomicAdd(&cnt[i], __popc(peers));
    }
}

// one block: the rows (seg_off) and 128-row units (unit_off) before each
// instance, count + 1 entries; cursor[i] = segment start for the scatter
__global__ void __launch_bounds__(1024) k_flag_units(const int *__restrict__ cnt, int count, int64_t *__restrict__ cursor,
                                                     int64_t *__restrict__ seg_off, int64_t *__restrict__ unit_off,
                                                     int *__restrict__ n_units) {
    __shared__ int64_t seg_carry, unit_carry;
    __shared__ int64_t s_seg[1024], s_unit[1024];
    if (threadIdx.x == 0) seg_carry = unit_carry = 0;
    __syncthreads();
    for (int base = 0; base < count; base += 1024) {
        const int i = base + threadIdx.x;
        const int64_t c = i < count ? cnt[i] : 0;
        const int64_t nu = (c + AS_TR - 1) / AS_TR;
        s_seg[threadIdx.x] = c;
        s_unit[threadIdx.x] = nu;
        __syncthreads();
        for (int o = 1; o < 1024 && o < count; o <<= 1) {  // inclusive scans
            const int64_t a = threadIdx.x >= o ? s_seg[threadIdx.x - o] : 0;
            const int64_t b = threadIdx.x >= o ? s_unit[threadIdx.x - o] : 0;
            __syncthreads();
            s_seg[threadIdx.x] += a;
            s_unit[threadIdx.x] += b;
            __syncthreads();
        }
        if (i < count) {
            cursor[i] = seg_off[i] = seg_carry + s_seg[threadIdx.x] - c;
            unit_off[i] = unit_carry + s_unit[threadIdx.x] - nu;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            const int last = min(1024, count - base) - 1;
            seg_carry += s_seg[last];
            unit_carry += s_unit[last];
        }
        __syncthreads();
    }
    if (threadIdx.x == 0) {
        seg_off[count] = seg_carry;
        unit_off[count] = unit_carry;
        *n_units = (int)unit_carry;
    }
}

// unit u: its instance, first row (in grows) and row count
__global__ void k_fill_units(int count, const int64_t *__restrict__ seg_off, const int64_t *__restrict__ unit_off,
                             int *__restrict__ unit_inst, int64_t *__restrict__ unit_start, int *__restrict__ unit_cnt) {
    const int64_t nu = unit_off[count];
    for (int64_t u = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; u < nu; u += (int64_t)gridDim.x * blockDim.x) {
        const int i = find_inst(unit_off, count, u);
        const int64_t s = seg_off[i] + (u - unit_off[i]) * AS_TR;
        unit_inst[u] = i;
        unit_start[u] = s;
        unit_cnt[u] = (int)min((int64_t)AS_TR, seg_off[i + 1] - s);
    }
}

__global__ void k_flag_scatter(const int32_t *__restrict__ flags, const unsigned long long *__restrict__ n_flag,
                               const int64_t *__restrict__ row_off, int count, int64_t *__restrict__ cursor,
                               int32_t *__restrict__ grows) {
    const int64_t nf = (int64_t)*n_flag;
    const int lane = threadIdx.x & 31;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q - lane < nf;
         q += (int64_t)gridDim.x * blockDim.x) {
        int32_t r;
        const int i = flag_inst(flags, q, nf, row_off, count, r);
        const uint32_t peers = __match_any_sync(0xffffffffu, i);
        const int first = __ffs(peers) - 1;
        unsigned long long at = 0;
        if (i >= 0 && lane == first) at = atomicAdd((unsigned long long *)&cursor[i], (unsigned long long)__popc(peers));
        at = __shfl_sync(0xffffffffu, at, first);
        if (i >= 0) grows[at + __popc(peers & ((1u << lane) - 1u))] = r;
    }
}

// Exact decision for flagged objects, one warp per object, one centre per
// lane (the row in shared memory): an FP32 pass over all centres finds the
// smallest fast value m; a second pass takes every centre whose fast value
// is within the FP32 window of m and decides among them with the FP64
// reference distance, ties to the smaller index.  Flag entries are global rows; instance i owns rows
// [row_off[i], row_off[i + 1]).  d <= 256.
// With flag_m, entry q brings the smallest fast value of its row from the
// tiled FP32 pass and the first pass is skipped.  Any fast value f' of any
// centre j' serves as m: the winner j* has fast(j*) <= D(j*) + W <= D(j') + W
// <= f' + 2W, W the rigorous FP32 window (both passes are within W of the
// exact distance whatever their summation order).  NaN: no finite value.
constexpr int RC_MAXD = 256;
__global__ void __launch_bounds__(256) k_assign_recheck(const RInst *__restrict__ R,
                                                        const int64_t *__restrict__ row_off, int count,
                                                        const int32_t *__restrict__ flag_rows,
                                                        const float *__restrict__ flag_m,
                                                        const unsigned long long *__restrict__ n_flag) {
    __shared__ __align__(16) float xs[8][RC_MAXD];  // the warp's row
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    const int64_t nf = (int64_t)*n_flag;
    for (int64_t q = warp; q < nf; q += nw) {
        const int64_t grow = flag_rows[q];
        const RInst &I = R[find_inst(row_off, count, grow)];
        const int64_t row = grow - I.row_base;
        const int d = I.d;
        const int64_t k = I.k;
        const float *xr = I.x + row * I.ldx;
        float xv[RC_MAXD / 32];
        float xs2 = 0.f;
#pragma unroll
        for (int u = 0; u < RC_MAXD / 32; u++) {
            const int t = lane + 32 * u;
            xv[u] = t < d ? xr[t] : 0.f;
            if (t < d) xs[wib][t] = xv[u];
            xs2 = fmaf(xv[u], xv[u], xs2);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) xs2 += __shfl_xor_sync(0xffffffffu, xs2, o);
        __syncwarp();
        const float xn = sqrtf(xs2) * (1.f + 1.0e-3f);
        const float cmax = __uint_as_float(*I.cmax_bits);
        // fast value of centre j, one centre per lane: the row is read from
        // shared memory (a broadcast), the centre from its own row
        const float *xw = xs[wib];
        const bool v4 = (d & 3) == 0 && (((uintptr_t)I.c32) & 15) == 0;
        auto fast = [&](int64_t j) {
            const float *cr = I.c32 + j * d;
            float dot = 0.f;
            if (v4) {
                for (int t = 0; t < d; t += 4) {
                    const float4 c4 = *reinterpret_cast<const float4 *>(cr + t);
                    const float4 x4 = *reinterpret_cast<const float4 *>(xw + t);
                    dot = fmaf(x4.x, c4.x, dot);
                    dot = fmaf(x4.y, c4.y, dot);
                    dot = fmaf(x4.z, c4.z, dot);
                    dot = fmaf(x4.w, c4.w, dot);
                }
            } else {
                for (int t = 0; t < d; t++) dot = fmaf(xw[t], cr[t], dot);
            }
            return fmaf(-2.f, dot, I.cn[j]);
        };
        float m = flag_m ? flag_m[q] : __int_as_float(0x7fc00000);
        if (m != m) {
            m = FLT_MAX;
            for (int64_t j0 = 0; j0 < k; j0 += 32) {
                const int64_t j = j0 + lane;
                if (j < k) m = fminf(m, fast(j));
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fminf(m, __shfl_xor_sync(0xffffffffu, m, o));
        }
        const float lim = m + 2.f * window_fp32(xn, cmax, d) * (1.f + 1e-6f);
        double bD = DBL_MAX;
        int bj = 0x7FFFFFFF;
        for (int64_t j0 = 0; j0 < k; j0 += 32) {
            const int64_t j = j0 + lane;
            // candidates: fast value within the window of m; the FP64
            // reference decides among them, each lane its own
            if (j < k && fast(j) <= lim) {
                const double D = ref_dist(xw, I.c64 + j * d, d);
                if (D < bD || (D == bD && (int)j < bj)) {
                    bD = D;
                    bj = (int)j;
                }
            }
        }
        // warp argmin, ties to the smaller index
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
            const double D2 = __shfl_xor_sync(0xffffffffu, bD, o);
            const int j2 = __shfl_xor_sync(0xffffffffu, bj, o);
            if (D2 < bD || (D2 == bD && j2 < bj)) {
                bD = D2;
                bj = j2;
            }
        }
        // no candidate with a distance below +inf (non-finite input): -1,
        // as the reference argmin that never improves on +inf
        if (lane == 0) I.labels[row] = bj == 0x7FFFFFFF ? -1 : bj;
        __syncwarp();
    }
}

// centre preparation: FP32 copy, |c|^2 (FP64 then rounded), max |c|.  A warp takes
// C.steps times a few centres, C.lanes lanes over each's coordinates; lane i then
// ends centre i.  What bounds many centres is FP64, two lanes per cycle and SM: a
// sum over 32 lanes and a square root for one centre cost as much as 300 and 600
// of its products (1M x 32: 185 us, with a warp per centre 1,014; 200,000 x 128: 137
// us, 277).  (A thread per centre took 26 us for 2,000 of 96 coordinates, now 4.5:
// scattered loads.)
template <class Inst>  // inst(e, j): the instance and local index of centre e
__device__ __forceinline__ void centre_prep(int64_t e0, int64_t ktot, CentreWarp C, Inst inst) {
    const int lane = threadIdx.x & 31, per = C.per_step();
    double mine = 0.0;
    for (int st = 0; st < C.steps; st++) {
        const int64_t e = e0 + per * st + lane / C.lanes;
        double s = 0.0;
        if (e < ktot) {
            int64_t j;
            const CInst &I = inst(e, j);
            const int d = I.d;
#pragma unroll 4
            for (int t = lane & (C.lanes - 1); t < d; t += C.lanes) {
                const double v = I.c64[j * d + t];
                I.c32[j * d + t] = (float)v;
                s += v * v;
            }
        }
        for (int o = 1; o < C.lanes; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        s = __shfl_sync(0xffffffffu, s, C.lanes * (lane & (per - 1)));
        if (lane / per == st) mine = s;
    }
    unsigned bits = 0;
    unsigned *most = nullptr;
    if (lane < C.centres() && e0 + lane < ktot) {
        int64_t j;
        const CInst &I = inst(e0 + lane, j);
        I.cn[j] = (float)mine;
        bits = __float_as_uint((float)sqrt(mine) * (1.f + 1e-6f));  // non-negative floats order as uints
        most = I.cmax_bits;
    }
    max_by_warp(most, bits);
}

// global centre e of instance find_inst(k_off, e)
__global__ void k_centre_prep(const CInst *__restrict__ C, const int64_t *__restrict__ k_off, int count,
                              int64_t ktot, CentreWarp W) {
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * W.centres() < ktot; w += nw)
        centre_prep(w * W.centres(), ktot, W, [&](int64_t e, int64_t &j) -> const CInst & {
            const CInst &I = C[find_inst(k_off, count, e)];
            j = e - I.k_base;
            return I;
        });
}

// one data set: its centres, and the one-instance tables of the kernels that
// read them from memory (one launch instead of four small copies)
struct OneTables {
    RInst r;
    int64_t row_off[2];
};
__global__ void k_centre_prep_one(const __grid_constant__ CInst I, int64_t k, CentreWarp W, OneTables T,
                                  OneTables *__restrict__ out) {
    if (blockIdx.x == 0 && threadIdx.x == 0) *out = T;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t w = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; w * W.centres() < k; w += nw)
        centre_prep(w * W.centres(), k, W, [&](int64_t e, int64_t &j) -> const CInst & {
            j = e;
            return I;
        });
}

// double-float split of the FP64 centres: c = hi + lo with hi = (float)c
__global__ void k_centre_split(const double *__restrict__ c64, int64_t kd, float *__restrict__ hi,
                               float *__restrict__ lo) {
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < kd; e += (int64_t)gridDim.x * blockDim.x) {
        const double c = c64[e];
        const float h = (float)c;
        hi[e] = h;
        lo[e] = (float)(c - (double)h);
    }
}

// running sum sh + sl of non-negative FP32 values with each addition's
// rounding error kept (TwoSum): relative error about 2^-23 for any count,
// in FP32 operations only
__device__ __forceinline__ void csum_add(float &sh, float &sl, float v) {
    const float t = __fadd_rn(sh, v);
    const float bb = __fsub_rn(t, sh);
    const float err = __fadd_rn(__fsub_rn(sh, __fsub_rn(t, bb)), __fsub_rn(v, bb));
    sh = t;
    sl = __fadd_rn(sl, err);
}

// Lane partials of four rows' distances to their labelled centres (rows
// i[q] < n; d <= 128, rows and centre halves 16-byte aligned): lane l holds
// coordinates 4l .. 4l+3, diff = (x - c_hi) - c_lo, squares summed in FP32.
// Every row's label and coordinates are requested before any centre, so the
// four rows' loads are in flight together.
__device__ __forceinline__ void dist4_vec(const float *__restrict__ x, int64_t ldx, int64_t n, int d,
                                          const float *__restrict__ chi, const float *__restrict__ clo, int64_t k,
                                          const int32_t *__restrict__ labels, const int64_t (&i)[4], float (&D)[4],
                                          bool (&ok)[4]) {
    const int lane = threadIdx.x & 31;
    const bool mine = 4 * lane < d;
    int j[4];
    float4 xv[4];
#pragma unroll
    for (int q = 0; q < 4; q++) {
        j[q] = i[q] < n ? labels[i[q]] : -1;
        xv[q] = (i[q] < n && mine) ? *reinterpret_cast<const float4 *>(x + i[q] * ldx + 4 * lane)
                                   : make_float4(0.f, 0.f, 0.f, 0.f);
    }
#pragma unroll
    for (int q = 0; q < 4; q++) {
        ok[q] = j[q] >= 0 && j[q] < k;  // uniform across the warp
        const bool use = ok[q] && mine;
        const float4 hv = use ? *reinterpret_cast<const float4 *>(chi + (int64_t)j[q] * d + 4 * lane)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
        const float4 lv = use ? *reinterpret_cast<const float4 *>(clo + (int64_t)j[q] * d + 4 * lane)
                              : make_float4(0.f, 0.f, 0.f, 0.f);
        const float e0 = (xv[q].x - hv.x) - lv.x, e1 = (xv[q].y - hv.y) - lv.y;
        const float e2 = (xv[q].z - hv.z) - lv.z, e3 = (xv[q].w - hv.w) - lv.w;
        D[q] = use ? fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, fmaf(e0, e0, 0.f)))) : 0.f;
    }
}

// per-object distance to its centre, warp per object, lanes over
// coordinates: diff = (x - c_hi) - c_lo, squares accumulated in FP32; the
// warp's distances in a compensated FP32 sum, block partial sums (FP64) and
// maxima, reduced on one block in a fixed order
__global__ void __launch_bounds__(256) k_assign_stats(const float *__restrict__ x, int64_t ldx, int64_t n, int d,
                                                      const float *__restrict__ chi, const float *__restrict__ clo,
                                                      int64_t k, const int32_t *__restrict__ labels,
                                                      double *__restrict__ part_sum, float *__restrict__ part_max) {
    __shared__ double ss[8];
    __shared__ float sm_[8];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    float sh = 0.f, sl = 0.f;  // compensated FP32 sum of the warp's distances
    float mx = 0.f;
    // rows, centre halves and the row pitch 16-byte aligned: a lane takes 4
    // consecutive coordinates per load (same summation depth per row)
    const bool vec = ((d & 3) == 0) && ((ldx & 3) == 0) && (((uintptr_t)x & 15) == 0) &&
                     (((uintptr_t)chi & 15) == 0) && (((uintptr_t)clo & 15) == 0);
    // four rows in flight per warp (independent loads and reductions)
    for (int64_t i0 = warp; i0 < n; i0 += 4 * nw) {
        float D[4];
        bool ok[4];
        if (vec && d <= 128) {
            const int64_t iq[4] = {i0, i0 + nw, i0 + 2 * nw, i0 + 3 * nw};
            dist4_vec(x, ldx, n, d, chi, clo, k, labels, iq, D, ok);
        } else {
#pragma unroll
        for (int q = 0; q < 4; q++) {
            const int64_t i = i0 + q * nw;
            const int j = i < n ? labels[i] : -1;
            ok[q] = j >= 0 && j < k;  // uniform across the warp
            D[q] = 0.f;
            if (ok[q]) {
                const float *xr = x + i * ldx;
                const float *h = chi + (int64_t)j * d;
                const float *l = clo + (int64_t)j * d;
                if (vec) {
                    for (int t = 4 * lane; t < d; t += 128) {
                        const float4 xv = *reinterpret_cast<const float4 *>(xr + t);
                        const float4 hv = *reinterpret_cast<const float4 *>(h + t);
                        const float4 lv = *reinterpret_cast<const float4 *>(l + t);
                        const float e0 = (xv.x - hv.x) - lv.x, e1 = (xv.y - hv.y) - lv.y;
                        const float e2 = (xv.z - hv.z) - lv.z, e3 = (xv.w - hv.w) - lv.w;
                        D[q] = fmaf(e3, e3, fmaf(e2, e2, fmaf(e1, e1, fmaf(e0, e0, D[q]))));
                    }
                } else {
                    for (int t = lane; t < d; t += 32) {
                        const float e = (xr[t] - h[t]) - l[t];
                        D[q] = fmaf(e, e, D[q]);
                    }
                }
            }
        }
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
            for (int q = 0; q < 4; q++) D[q] += __shfl_xor_sync(0xffffffffu, D[q], o);
        }
#pragma unroll
        for (int q = 0; q < 4; q++)
            if (ok[q]) {
                csum_add(sh, sl, D[q]);
                mx = fmaxf(mx, D[q]);
            }
    }
    if (lane == 0) {
        ss[wib] = (double)sh + (double)sl;
        sm_[wib] = mx;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0;
        float m = 0.f;
        for (int w = 0; w < 8; w++) {
            a += ss[w];
            m = fmaxf(m, sm_[w]);
        }
        part_sum[blockIdx.x] = a;
        part_max[blockIdx.x] = m;
    }
}

// one block: the block partials in a fixed order (thread t takes partials t, t +
// 256, ..., then a tree); a single thread took 0.25 ms for 4,864 of them
__global__ void __launch_bounds__(256) k_stats_final(const double *__restrict__ ps, const float *__restrict__ pm, int nb,
                                                     double *__restrict__ out) {
    __shared__ double ss[256];
    __shared__ float sx[256];
    const int t = threadIdx.x;
    double s = 0.0;
    float m = 0.f;
    for (int i = t; i < nb; i += 256) {
        s += ps[i];
        m = fmaxf(m, pm[i]);
    }
    ss[t] = s;
    sx[t] = m;
    for (int o = 128; o > 0; o >>= 1) {
        __syncthreads();
        if (t < o) {
            ss[t] += ss[t + o];
            sx[t] = fmaxf(sx[t], sx[t + o]);
        }
    }
    if (t == 0) {
        out[0] = ss[0];
        out[1] = sqrt((double)sx[0]);
    }
}

// centroid coordinate t of the seed with members sids[s0 .. s1) (ascending
// ids, rows x + (id - row_base) * ldx): FP64 sum in member order, one IEEE
// division by the count
__device__ __forceinline__ double centroid_coord(const float *__restrict__ x, int64_t ldx, int64_t row_base,
                                                 const int32_t *__restrict__ sids, int64_t s0, int64_t s1, int t) {
    double s = 0.0;
    for (int64_t p = s0; p < s1; p++) s = __dadd_rn(s, (double)x[((int64_t)sids[p] - row_base) * ldx + t]);
    return __ddiv_rn(s, (double)(s1 - s0));
}

// centroid of each seed; one thread per (seed, coordinate)
__global__ void k_centroids(const float *__restrict__ x, int64_t ldx, int d, int64_t k,
                            const int64_t *__restrict__ soff, const int32_t *__restrict__ sids,
                            double *__restrict__ c) {
    const int64_t total = k * d;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t j = e / d;
        const int t = (int)(e % d);
        c[e] = centroid_coord(x, ldx, 0, sids, soff[j], soff[j + 1], t);
    }
}

// batched: thread per (global seed, coordinate < dmax); instance i owns
// seeds [seed_inst_off[i], seed_inst_off[i + 1])
__global__ void k_centroids_batch(const CenInst *__restrict__ C, const int64_t *__restrict__ seed_inst_off,
                                  int count, int64_t ktot, int dmax, const int64_t *__restrict__ soff,
                                  const int32_t *__restrict__ sids) {
    const int64_t total = ktot * dmax;
    for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < total;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int64_t s = e / dmax;
        const int t = (int)(e % dmax);
        const CenInst &I = C[find_inst(seed_inst_off, count, s)];
        if (t >= I.d) continue;
        I.c[(s - I.seed_base) * I.d + t] = centroid_coord(I.x, I.ldx, I.row_base, sids, soff[s], soff[s + 1], t);
    }
}

// batched SSE / radius partials: block per 128-row unit (instance, tile),
// warp per row, squares of (x - c_hi) - c_lo accumulated in FP32
__global__ void __launch_bounds__(256, 4) k_assign_stats_batch(const SInst *__restrict__ S, const int2 *__restrict__ units,
                                                            int64_t nunits, double *__restrict__ part_sum,
                                                            float *__restrict__ part_max) {
    __shared__ double ss[8];
    __shared__ float sm_[8];
    const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
    for (int64_t u = blockIdx.x; u < nunits; u += gridDim.x) {
        const int2 un = units[u];
        const SInst &I = S[un.x];
        float sh = 0.f, sl = 0.f;  // compensated FP32 sum of the warp's distances
        float mx = 0.f;
        const bool vec = I.d <= 128 && ((I.d & 3) == 0) && ((I.ldx & 3) == 0) && (((uintptr_t)I.x & 15) == 0) &&
                         (((uintptr_t)I.chi & 15) == 0) && (((uintptr_t)I.clo & 15) == 0);
        // rows wib, wib + 8, ... of the unit, four in flight per warp
        for (int r0 = wib; r0 < 128; r0 += 32) {
            float D[4];
            bool ok[4];
            if (vec) {
                const int64_t b = (int64_t)un.y * 128 + r0;
                const int64_t iq[4] = {b, b + 8, b + 16, b + 24};
                dist4_vec(I.x, I.ldx, I.n, I.d, I.chi, I.clo, I.k, I.labels, iq, D, ok);
            } else {
#pragma unroll
            for (int q = 0; q < 4; q++) {
                const int64_t i = (int64_t)un.y * 128 + r0 + 8 * q;
                const int j = i < I.n ? I.labels[i] : -1;
                ok[q] = j >= 0 && j < I.k;  // uniform across the warp
                D[q] = 0.f;
                if (ok[q]) {
                    const float *xr = I.x + i * I.ldx;
                    const float *h = I.chi + (int64_t)j * I.d;
                    const float *l = I.clo + (int64_t)j * I.d;
                    for (int t = lane; t < I.d; t += 32) {
                        const float e = (xr[t] - h[t]) - l[t];
                        D[q] = fmaf(e, e, D[q]);
                    }
                }
            }
            }
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
                for (int q = 0; q < 4; q++) D[q] += __shfl_xor_sync(0xffffffffu, D[q], o);
            }
#pragma unroll
            for (int q = 0; q < 4; q++)
                if (ok[q]) {
                    csum_add(sh, sl, D[q]);
                    mx = fmaxf(mx, D[q]);
                }
        }
        __syncthreads();
        if (lane == 0) {
            ss[wib] = (double)sh + (double)sl;
            sm_[wib] = mx;
        }
        __syncthreads();
        if (threadIdx.x == 0) {
            double a = 0.0;
            float m = 0.f;
            for (int w = 0; w < 8; w++) {
                a += ss[w];
                m = fmaxf(m, sm_[w]);
            }
            part_sum[u] = a;
            part_max[u] = m;
        }
    }
}

// Per-cluster radius (Sect. 4.1): for every object its distance to its
// centre as in k_assign_stats (warp per object, diff = (x - c_hi) - c_lo,
// squares in FP32), and per label the largest one by an atomic maximum on the
// bits of the non-negative float.
__global__ void __launch_bounds__(256) k_cluster_rmax(const float *__restrict__ x, int64_t ldx, int64_t n, int d,
                                                      const float *__restrict__ chi, const float *__restrict__ clo,
                                                      int64_t k, const int32_t *__restrict__ labels,
                                                      unsigned *__restrict__ rmax) {
    const int lane = threadIdx.x & 31;
    const int64_t warp = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t i = warp; i < n; i += nw) {
        const int j = labels[i];
        if (j < 0 || j >= k) continue;  // warp-uniform
        const float *xr = x + i * ldx;
        const float *h = chi + (int64_t)j * d;
        const float *l = clo + (int64_t)j * d;
        float D = 0.f;
        for (int t = lane; t < d; t += 32) {
            const float e = (xr[t] - h[t]) - l[t];
            D = fmaf(e, e, D);
        }
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) D += __shfl_xor_sync(0xffffffffu, D, o);
        if (lane == 0) atomicMax(&rmax[j], __float_as_uint(D));
    }
}

__global__ void k_cluster_sqrt(int64_t k, const unsigned *__restrict__ rmax, double *__restrict__ radius) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < k; j += (int64_t)gridDim.x * blockDim.x)
        radius[j] = sqrt((double)__uint_as_float(rmax[j]));
}

// per instance: its units' partials in unit order (deterministic)
__global__ void k_stats_final_batch(const double *__restrict__ ps, const float *__restrict__ pm,
                                    const int64_t *__restrict__ unit_off, int count, double *__restrict__ sse,
                                    double *__restrict__ rmax) {
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < count; i += gridDim.x * blockDim.x) {
        double s = 0.0;
        float m = 0.f;
        for (int64_t u = unit_off[i]; u < unit_off[i + 1]; u++) {
            s += ps[u];
            m = fmaxf(m, pm[u]);
        }
        sse[i] = s;
        rmax[i] = sqrt((double)m);
    }
}

__global__ void k_fill_labels(int32_t *l, int64_t n, int32_t v) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        l[i] = v;
}

}  // namespace

geek_status centroids_from_seeds(geek_ctx *ctx, const float *x, int64_t ldx, int d, const silk_seeds *s,
                                 double *centres, cudaStream_t st) {
    if (s->k == 0) return GEEK_OK;
    GK_COUNT();
    k_centroids<<<grid_for(s->k * d, 256, ctx->num_sms), 256, 0, st>>>(x, ldx, d, s->k, s->off, s->ids, centres);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

// ---- extra passes of assignment (Sect. 5) --------------------------------
// members grouped by label: key = label (k for -1), id; counts per label
__global__ void k_label_keys(int64_t n, const int32_t *__restrict__ labels, int64_t k, uint64_t *__restrict__ key,
                             uint32_t *__restrict__ ids, unsigned long long *__restrict__ cnt, int *__restrict__ bad) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        int64_t l = labels[i];
        if (l < -1 || l >= k) {
            atomicExch(bad, 1);
            l = -1;
        }
        key[i] = l < 0 ? (uint64_t)k : (uint64_t)l;
        ids[i] = (uint32_t)i;
        if (l >= 0) atomicAdd(&cnt[l], 1ull);
    }
}

// sort key of centre j: descending member count, then ascending index; nseg[j] = 0
__global__ void k_size_order(int64_t k, const unsigned long long *__restrict__ cnt, uint64_t *__restrict__ key,
                             int64_t *__restrict__ nseg) {
    for (int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; j < k; j += (int64_t)gridDim.x * blockDim.x) {
        const uint64_t cj = cnt[j] > 0xFFFFFFFFull ? 0xFFFFFFFFull : cnt[j];
        key[j] = ((0xFFFFFFFFull - cj) << 32) | (uint64_t)j;
        nseg[j] = 0;
    }
}

// How many of the centres, the largest first, are cut into segments (the large
// ones): *n_large, and their segments in nseg.  Estimated, in ms, for every count
// (block of one):
//  the others' chains, 41 ns per member: the longest of them, or their balanced load
//  on the warp pairs;
//  the large ones' segments: two passes over their rows, 0.1 + 5.2 ps per value, and a
//  walk that grows as the root of the longest chain (most of its steps are near the
//  start), 0.1 + a sqrt(members / 1000), a = 0.11 with 32 coordinates per warp, 0.04
//  with 8.  It depends on the data (spread 1 around 10: up to 1.5 times that, around
//  100: down to 0.7) and is taken for 1.25 times that where the others' chains follow
//  it, for 0.55 where they run beside the walk: a chain left beside a short walk
//  costs more than a segment too many.
// Measured, chains and segments: 60 clusters of 20,000 x 128 0.82 and 2.6 ms, 20 of
// 50,000 1.9 and 2.4, 8 of 80,000 3.1 and 2.1, one of 20,000 0.77 and 0.73, one of
// 250,000 9.7 and 2.4; 111,000 x 128 of 105 Zipf clusters, one above UL_MIN, two
// passes 2.3 and 3.1 in all; 10M x 128 of 20,000 Zipf clusters 14 ms as chosen, 16
// with all above UL_MIN cut.
constexpr int UL_M = 128;        // members per segment
constexpr int UL_MIN = 16384;    // no smaller centre is large
__global__ void __launch_bounds__(256) k_large(int64_t k, int64_t most_large, int64_t n, int d, int pairs, bool beside,
                                               const unsigned long long *__restrict__ cnt,
                                               const uint64_t *__restrict__ order, int64_t *__restrict__ nseg,
                                               unsigned long long *__restrict__ n_large) {
    __shared__ unsigned long long s_best;
    __shared__ double s_warp[8];
    const int t = threadIdx.x, lane = t & 31, w = t >> 5;
    auto size = [&](int64_t q) { return q < k ? (double)cnt[order[q] & 0xFFFFFFFFull] : 0.0; };
    auto chains = [&](double longest, double rows) {
        return 41e-6 * fmax(longest, rows * d / (32.0 * pairs));
    };
    const double first = size(0);
    const double walk = (beside ? 0.55 : 1.25) * (0.1 + (0.02 + 0.09 * min(d, 32) / 32) * sqrt(first * 1e-3));
    // (estimate, count) of the best: positive floats order as their bits
    if (t == 0) s_best = (unsigned long long)__float_as_uint((float)chains(first, (double)n)) << 32;
    __syncthreads();
    double before = 0.0;
    for (int64_t q0 = 0; q0 < most_large; q0 += 256) {
        const int64_t q = q0 + t;
        const double c = q < most_large ? size(q) : 0.0, next = size(q + 1);
        double x = c > UL_MIN ? c : 0.0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const double y = __shfl_up_sync(0xffffffffu, x, o);
            if (lane >= o) x += y;
        }
        if (lane == 31) s_warp[w] = x;
        __syncthreads();
        double all = 0.0;
        for (int v = 0; v < 8; v++) {
            if (v < w) x += s_warp[v];
            all += s_warp[v];
        }
        if (c > UL_MIN) {  // the first q + 1
            const double rows = before + x;
            const double passes = 1.25 * (0.1 + 5.2e-9 * rows * d), rest = chains(next, (double)n - rows);
            const float est = (float)(passes + (beside ? fmax(walk, rest) : walk + rest));
            atomicMin(&s_best, ((unsigned long long)__float_as_uint(est) << 32) | (unsigned long long)(q + 1));
        }
        before += all;
        if (__syncthreads_or(c <= UL_MIN)) break;  // descending
    }
    __syncthreads();
    const int64_t nl = (int64_t)(s_best & 0xFFFFFFFFull);
    for (int64_t q = t; q < nl; q += 256) {
        const int64_t j = (int64_t)(order[q] & 0xFFFFFFFFull);
        nseg[j] = (int64_t)((cnt[j] + UL_M - 1) / UL_M);
    }
    if (t == 0) *n_large = (unsigned long long)nl;
}

// centre j <- mean of its members (ascending id, the seeds' centroid sum);
// no member: unchanged.  Work item = (centre, slice of 32 coordinates), one
// warp per item, lane = coordinate; each lane's sum is the sequential FP64
// chain s <- RN(s + x_i) over the centre's members in ascending id.
//
// An FP64 add on this part takes 60-170 cycles in a dependent chain (longer
// for operands of mixed exponents), which would bound the pass by the
// largest cluster's member count times that latency.  So each 32-member
// chunk first runs the chain in 64-bit integers, in a unit 2^g that divides
// s and every x_i of the chunk (the finer of s's lowest set bit and the
// finest ulp among the x_i): s = T 2^g.  While every partial sum T + R_1 +
// ... + R_i (R_i = x_i / 2^g) stays below 2^53 in magnitude, each partial
// sum is exactly representable in FP64, so each RN step is exact and the
// chain equals the integer sum (binade and sign changes included).  The
// first step that breaks this (a sum reaching 2^53 units, where rounding may
// start; an x_i too far above the unit or not finite), and every step after
// it in the chunk, runs as the FP64 add itself; so the result is the FP64
// chain bit for bit.  The integer sum is accumulated unconditionally (a
// 64-bit add is the only loop-carried step) and the failures collected in a
// bit mask.
//
// Each work item is served by a pair of warps: a producer (fetches the item,
// loads the member ids four stages ahead, copies 32 member rows per stage
// into the pair's ring of UC_S stages with 16-byte cp.async, 4 rows per
// instruction) and a consumer (the chain above, a stage at a time), so the
// consumer's single instruction stream carries only the sums.  Stage hand-off
// by mbarriers: "full" completes when the producer's 32 lanes' copies have
// landed (cp.async.mbarrier.arrive.noinc) and its header is written, "empty"
// when the consumer is done with the stage; every wait is bounded (on expiry
// the kernel records GEEK_ERR_TIMEOUT and both warps stop).  The first wave of
// items goes to pairs pair-in-block major, so the slices of one centre start
// on different SMs; later items come from an atomic counter, largest centre
// first (order: centre indices by descending member count).
constexpr int UC_P = 4, UC_T = 64 * UC_P, UC_B = 32, UC_S = 8;
constexpr int UC_STAGE = UC_B * 32;                                    // floats per stage
constexpr int UC_SMEM = UC_P * UC_S * UC_STAGE * (int)sizeof(float);   // 128 KB of rings

// a stage's header: which item and which 32 members
struct UcHdr {
    int64_t j, cj;  // centre, its member count (cj < 0: no more items)
    int32_t t0, g;  // first coordinate of the slice, member group
};

// x / 2^g as a signed integer, x = +-mx 2^u with base = 150 + g and u >= g:
// exact for u - g <= 38 (then |x / 2^g| < 2^62); bad beyond that or when x
// is not finite
__device__ __forceinline__ int64_t units_of(float x, int base, bool &bad) {
    const uint32_t b = __float_as_uint(x);
    const int e = (int)((b >> 23) & 0xFFu);
    const uint32_t mx = (b & 0x7FFFFFu) | ((uint32_t)min(e, 1) << 23);
    const int lsh = max(e, 1) - base;  // u - g >= 0
    bad = lsh > 38 || e == 0xFF;
    const int64_t R = (int64_t)((uint64_t)mx << (lsh & 63));
    return (b >> 31) ? -R : R;
}

// s <- RN(...RN(RN(s + v[0]) + v[1]) ... + v[ma - 1]) in FP64, ma <= 32 (a
// lane with act = false, past the last coordinate, takes no FP64 step and
// so holds up no other lane)
// FULL: ma == UC_B, every step unpredicated and the one-check sum a tree.
template <bool FULL>
__device__ __forceinline__ double chain_chunk(double s, const float (&v)[UC_B], int ma, bool act) {
    if (FULL) ma = UC_B;
    constexpr uint64_t M52 = (1ull << 52) - 1;
    const uint64_t bits = (uint64_t)__double_as_longlong(s);
    const int E = (int)((bits >> 52) & 0x7FF);
    const bool zero = bits == 0;  // +0 (the running sum never becomes -0)
    // integer steps from +0 or from a normal s well inside the range
    bool fast = zero || (E > 64 && E < 0x7FE - 64);
    const uint64_t M = (bits & M52) | (1ull << 52);
    // the unit 2^g: the finest ulp among the chunk's values and s's lowest set bit
    // (tree reductions: no 32-long dependency chain)
    int ua[UC_B], ea[UC_B];
#pragma unroll
    for (int m = 0; m < UC_B; m++) {
        const int e = (int)((__float_as_uint(v[m]) >> 23) & 0xFFu);
        ua[m] = m < ma ? max(e, 1) : 0x7FFFFFFF;
        ea[m] = m < ma ? e : 0;
    }
#pragma unroll
    for (int w = 1; w < UC_B; w <<= 1)
#pragma unroll
        for (int m = 0; m < UC_B; m += 2 * w) {
            ua[m] = min(ua[m], ua[m + w]);
            ea[m] = max(ea[m], ea[m + w]);
        }
    const int umin = ua[0], emax = ea[0];
    const int qs = E - 1075;
    const int g = zero ? umin - 150 : min(umin - 150, qs + __ffsll((long long)M) - 1);
    int64_t T0 = 0;
    if (!zero) {
        const int sh = qs - g;  // > 0: s's ulp is coarser than a value's (s then needs more than 53 bits)
        fast = fast && sh <= 10;
        const uint64_t a0 = sh >= 0 ? (M << min(sh, 10)) : (M >> min(-sh, 63));  // exact: g <= s's lowest set bit
        T0 = (bits >> 63) ? -(int64_t)a0 : (int64_t)a0;
    }
    const int base = 150 + g;
    // every |x_i / 2^g| < 2^(24 + lmax) (0 <= lmax): if |T0| + 32 2^(24 + lmax)
    // < 2^53, no partial sum can reach 2^53 and the chunk is one exact
    // integer sum (any order); otherwise each partial sum is checked
    const int lmax = max(emax, 1) - base;
    const uint64_t aT0 = (uint64_t)(T0 < 0 ? -T0 : T0);
    const bool easy = fast && emax != 0xFF && lmax <= 23 && aT0 + (1ull << (29 + lmax)) < (1ull << 53);
    int64_t T = T0;
    int f = ma;  // first step that takes the FP64 add
    if (easy && FULL) {
        int64_t r[UC_B];
#pragma unroll
        for (int m = 0; m < UC_B; m++) {
            bool bad;
            r[m] = units_of(v[m], base, bad);
        }
#pragma unroll
        for (int w = 1; w < UC_B; w <<= 1)
#pragma unroll
            for (int m = 0; m < UC_B; m += 2 * w) r[m] += r[m + w];
        T += r[0];
    } else if (easy) {
        int64_t p1 = 0, p2 = 0, p3 = 0;
#pragma unroll
        for (int m = 0; m < UC_B; m += 4) {
            bool bad;
            if (m < ma) T += units_of(v[m], base, bad);
            if (m + 1 < ma) p1 += units_of(v[m + 1], base, bad);
            if (m + 2 < ma) p2 += units_of(v[m + 2], base, bad);
            if (m + 3 < ma) p3 += units_of(v[m + 3], base, bad);
        }
        T += p1 + p2 + p3;
    } else if (act) {
        uint32_t fail = fast ? 0u : 1u;
#pragma unroll
        for (int m = 0; m < UC_B; m++) {
            if (m < ma) {
                bool bad;
                T += units_of(v[m], base, bad);
                // |T| < 2^53: every partial sum is an FP64 value, each RN step exact
                const bool ok = !bad && (uint64_t)(T + (int64_t)((1ull << 53) - 1)) < (1ull << 54) - 1;
                if (!ok) fail |= 1u << m;
            }
        }
        f = fail ? __ffs((int)fail) - 1 : ma;
    }
    if (f < ma && f > 0) {  // the integer sum up to step f - 1
        T = T0;
#pragma unroll
        for (int m = 0; m < UC_B; m++)
            if (m < f) {
                bool bad;
                T += units_of(v[m], base, bad);
            }
    }
    double t = s;
    if (f > 0 && act) {  // T 2^g, |T| < 2^53, as an FP64 value (exact)
        const uint64_t a = (uint64_t)(T < 0 ? -T : T);
        if (a == 0) {
            t = 0.0;  // an exactly cancelling sum is +0 under RN
        } else {
            const int p = 64 - __clzll((long long)a);  // <= 53
            const uint64_t mant = (a << (53 - p)) & M52;
            t = __longlong_as_double(
                (long long)(((uint64_t)(T < 0) << 63) | ((uint64_t)(g + 1075 + p - 53) << 52) | mant));
        }
    }
    if (__all_sync(0xffffffffu, f >= ma)) return t;
    const int fw = __reduce_min_sync(0xffffffffu, f);  // warp-uniform bound of the FP64 tail
#pragma unroll
    for (int m = 0; m < UC_B; m++)
        if (m >= fw && m < ma && m >= f) t = __dadd_rn(t, widen_f32(v[m]));
    return t;
}

__device__ __forceinline__ void cp_async16(uint32_t dst, const void *src, int bytes) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void cp_async4(uint32_t dst, const void *src, int bytes) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(dst), "l"(src), "r"(bytes) : "memory");
}

__device__ __forceinline__ void cp_async_bar_arrive(uint64_t *bar) {
    asm volatile("cp.async.mbarrier.arrive.noinc.shared::cta.b64 [%0];" ::"r"(su32(bar)) : "memory");
}

__global__ void __launch_bounds__(UC_T) k_update_centres(const float *__restrict__ x, int64_t ldx, int d, int64_t k,
                                                         const int64_t *__restrict__ off,
                                                         const unsigned long long *__restrict__ cnt,
                                                         const int32_t *__restrict__ ids, const uint64_t *__restrict__ order,
                                                         const unsigned long long *__restrict__ n_large,
                                                         unsigned long long *__restrict__ next, double *__restrict__ c,
                                                         int *__restrict__ err) {
    extern __shared__ float uc_ring[];  // [UC_P][UC_S][32 rows][32 floats]
    __shared__ UcHdr hdr[UC_P][UC_S];
    __shared__ uint64_t full[UC_P][UC_S], empty[UC_P][UC_S];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool producer = warp >= UC_P;
    const int pr = producer ? warp - UC_P : warp;  // the pair
    float *ring = uc_ring + (size_t)pr * UC_S * UC_STAGE;
    if (threadIdx.x < UC_P * UC_S) {
        mbar_init(&full[threadIdx.x / UC_S][threadIdx.x % UC_S], 33);  // 32 copy arrivals + the header
        mbar_init(&empty[threadIdx.x / UC_S][threadIdx.x % UC_S], 1);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    __syncthreads();
    const int nsl = (d + 31) >> 5;
    const int64_t nitems = k * nsl;
    if (producer) {
        const uint32_t ring_s = su32(ring);
        const bool vec = (((uintptr_t)x & 15) == 0) && ((ldx & 3) == 0);
        const int64_t np = (int64_t)gridDim.x * UC_P;
        const int64_t it0 = (int64_t)*n_large * nsl;        // the large centres come first in the order
        int64_t it = it0 + (int64_t)pr * gridDim.x + blockIdx.x;  // first wave: slices of a centre on different SMs
        uint32_t sn = 0;                                    // stages issued by this pair
        bool ok = true;
        for (;;) {
            const bool done = it >= nitems;
            int64_t j = 0, cj = 0;
            int t0 = 0;
            if (!done) {
                j = (int64_t)(order[it / nsl] & 0xFFFFFFFFull);
                t0 = (int)(it % nsl) * 32;
                cj = (int64_t)cnt[j];
            }
            const int width = min(32, d - t0);
            const int col = (lane & 7) * 4;  // this lane's 16 bytes of a row slice (vector copies)
            const int nbytes = max(0, min(16, (width - col) * 4));
            const int32_t *mid = ids + (done ? 0 : off[j]);
            const float *xs = x + t0;
            const int64_t ng = done ? 1 : (cj + UC_B - 1) / UC_B;  // the end marker takes one stage
            auto ld_id = [&](int64_t g) -> int32_t {
                const int64_t q = g * UC_B + lane;
                return (!done && q < cj) ? mid[q] : 0;
            };
            int32_t id0 = ld_id(0), id1 = ld_id(1), id2 = ld_id(2), id3 = ld_id(3);
            for (int64_t g = 0; g < ng && ok; g++, sn++) {
                const int st = (int)(sn % UC_S);
                const uint32_t use = sn / UC_S;
                if (lane == 0) ok = mbar_wait(&empty[pr][st], (use & 1) ^ 1, err);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) break;
                const int32_t my = id0;
                id0 = id1;
                id1 = id2;
                id2 = id3;
                id3 = ld_id(g + 4);
                if (!done) {
                    const int rows = (int)min((int64_t)UC_B, cj - g * UC_B);
                    const uint32_t sb = ring_s + (uint32_t)(st * UC_STAGE * sizeof(float));
                    if (vec) {
#pragma unroll
                        for (int i = 0; i < UC_B / 4; i++) {
                            const int rr = 4 * i + (lane >> 3);
                            const int32_t r = __shfl_sync(0xffffffffu, my, rr);
                            if (rr < rows)
                                cp_async16(sb + (uint32_t)(rr * 32 + col) * 4u, xs + (int64_t)r * ldx + (nbytes ? col : 0),
                                           nbytes);
                        }
                    } else {
#pragma unroll 8
                        for (int rr = 0; rr < UC_B; rr++) {
                            const int32_t r = __shfl_sync(0xffffffffu, my, rr);
                            if (rr < rows)
                                cp_async4(sb + (uint32_t)(rr * 32 + lane) * 4u, xs + (int64_t)r * ldx + (lane < width ? lane : 0),
                                          lane < width ? 4 : 0);
                        }
                    }
                }
                cp_async_bar_arrive(&full[pr][st]);  // when this lane's copies have landed
                if (lane == 0) {
                    hdr[pr][st] = UcHdr{j, done ? -1 : cj, t0, (int32_t)g};
                    mbar_arrive(&full[pr][st]);
                }
            }
            if (done || !ok) break;
            unsigned long long got = 0;
            if (lane == 0) got = atomicAdd(next, 1ull);
            it = it0 + np + (int64_t)__shfl_sync(0xffffffffu, got, 0);
        }
        asm volatile("cp.async.wait_all;" ::: "memory");  // own copies landed before the block ends
    } else {
        double s = 0.0;
        for (uint32_t sn = 0;; sn++) {
            const int st = (int)(sn % UC_S);
            const uint32_t use = sn / UC_S;
            // lane 0 waits; __syncwarp then orders the other lanes' reads after
            // its acquire of the phase (the copies were the producer's)
            int okw = 0;
            if (lane == 0) okw = mbar_wait(&full[pr][st], use & 1, err);
            okw = __shfl_sync(0xffffffffu, okw, 0);
            __syncwarp();
            if (!okw) break;
            const UcHdr h = hdr[pr][st];
            if (h.cj < 0) break;
            const int width = min(32, d - h.t0);
            if (h.g == 0) s = 0.0;
            const float *src = ring + st * UC_STAGE + lane;
            float v[UC_B];
#pragma unroll
            for (int m = 0; m < UC_B; m++) v[m] = src[m * 32];
            const int ma = (int)min((int64_t)UC_B, h.cj - (int64_t)h.g * UC_B);
            s = ma == UC_B ? chain_chunk<true>(s, v, ma, lane < width) : chain_chunk<false>(s, v, ma, lane < width);
            __syncwarp();  // every lane's reads done before the stage is refilled
            if (lane == 0) mbar_arrive(&empty[pr][st]);
            if ((int64_t)(h.g + 1) * UC_B >= h.cj && lane < width) c[h.j * d + h.t0 + lane] = __ddiv_rn(s, (double)h.cj);
        }
    }
}

// ---- large centres: the chain in parallel segments -------------------------
// One warp walks a chain at about 42 ns per member, so a cluster of 950,000
// members held the whole pass for 38 ms (10M x 128, k = 20,000 with Zipf
// weights).  The chain s <- RN(s + x_i) can be cut into segments of UL_M
// members that run in parallel, bit for bit:
//  While s stays inside one binade, |s| in [2^e, 2^(e+1)), every FP64 value
//  there is a multiple of q = 2^(e-52), and RN(s + x) = s + q round(x / q) with
//  the ties of x / q broken by the parity of s / q.  So a whole segment moves
//  S = s / q by an integer that depends on S only through its parity: two
//  integers (for S even and odd) describe it, computed without knowing s, only
//  its binade.  The binade comes from the segments' approximate sums.
//  k_ul_sums    approximate sum of every (segment, coordinate), in a
//               compensated FP32 sum
//  k_ul_starts  their running sums: the approximate s at each segment's start
//  k_ul_deltas  the segment's two integers in the unit of that s's binade, and
//               the range of the partial sums on the way
//  k_ul_chain   a warp per (centre, 32 coordinates) walks the segments with the
//               exact s: where s has the assumed exponent and S plus the range
//               stays in [2^52 + 1, 2^53 - 1] (then every exact s + x lies in
//               the binade before its rounding), s moves by the integer;
//               otherwise (the first segments, a segment that crosses a power
//               of two, a member comparable to s or not finite) the segment
//               runs through chain_chunk.
// Which centres are cut: k_large.
struct UlArgs {
    const float *x;
    int64_t ldx;
    int d;
    int64_t k;
    const int64_t *off;
    const unsigned long long *cnt;
    const int32_t *ids;
    const int64_t *seg_off;        // k: first segment of each centre
    const int64_t *n_seg;          // all segments
    const uint64_t *order;         // centres by descending count
    const unsigned long long *n_large;
    double *start;                 // [segment][d]: sums, then s at the start (approximate)
    int64_t *rec;                  // [3][segments][d], see ul_pack
    int64_t segs;                  // segments the arrays hold
    double *c;                     // k x d
};

// A segment's three words for one coordinate: (D0, D1 - D0 + 1), (mn, low
// exponent bits), (mx, high exponent bits; 7: not usable).  D1 - D0 is -1, 0
// or 1 (rounding is monotone, so neighbours stay ordered, and they merge when
// both round to the same even value), and the three integers are below 2^54
// whenever the segment is usable.
__device__ __forceinline__ void ul_pack(int64_t *w, int64_t stride, int64_t D0, int64_t D1, int64_t mn, int64_t mx, int E,
                                        bool ok) {
    constexpr int64_t LIM = 1ll << 54;
    ok = ok && mn > -LIM && mx < LIM;
    w[0] = ok ? D0 * 4 + (D1 - D0 + 1) : 0;
    w[stride] = ok ? mn * 256 + (E & 0xFF) : 0;
    w[2 * stride] = ok ? mx * 256 + (E >> 8) : 7;
}

// item (segment, 32-coordinate slice) -> centre, member range, coordinate
struct UlItem {
    int64_t j, seg;
    const int32_t *mid;
    int rows, t;
    bool act;
};
__device__ __forceinline__ UlItem ul_item(const UlArgs &A, int64_t it, int nsl) {
    UlItem q;
    q.seg = it / nsl;
    q.t = (int)(it % nsl) * 32 + (threadIdx.x & 31);
    q.act = q.t < A.d;
    q.j = find_inst(A.seg_off, (int)A.k, q.seg);  // centres without segments share their successor's offset
    const int64_t m0 = (q.seg - A.seg_off[q.j]) * UL_M;
    q.rows = (int)min((int64_t)UL_M, (int64_t)A.cnt[q.j] - m0);
    q.mid = A.ids + A.off[q.j] + m0;
    return q;
}

// calls f(x) for the item's members in order, UL_F rows' loads in flight
constexpr int UL_F = 16;
template <class Fn>
__device__ __forceinline__ void ul_rows(const UlArgs &A, const UlItem &q, Fn f) {
    const int lane = threadIdx.x & 31;
    const float *xs = A.x + (q.act ? q.t : 0);
    for (int m0 = 0; m0 < q.rows; m0 += 32) {
        const int32_t id = m0 + lane < q.rows ? q.mid[m0 + lane] : 0;
        const int nr = min(32, q.rows - m0);
#pragma unroll
        for (int h = 0; h < 32; h += UL_F) {
            float v[UL_F];
#pragma unroll
            for (int r = 0; r < UL_F; r++) {
                const int32_t row = __shfl_sync(0xffffffffu, id, h + r);
                v[r] = h + r < nr ? xs[(int64_t)row * A.ldx] : 0.f;
            }
#pragma unroll
            for (int r = 0; r < UL_F; r++)
                if (h + r < nr) f(v[r]);
        }
    }
}

__global__ void __launch_bounds__(256) k_ul_sums(UlArgs A) {
    const int nsl = (A.d + 31) >> 5;
    const int64_t items = *A.n_seg * nsl, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += nw) {
        const UlItem q = ul_item(A, it, nsl);
        float sh = 0.f, sl = 0.f;
        ul_rows(A, q, [&](float v) { csum_add(sh, sl, v); });
        if (q.act) A.start[q.seg * A.d + q.t] = (double)sh + (double)sl;
    }
}

// block per (large centre, slice): sums -> the running sum before each segment;
// each of the 8 warps takes an eighth of the segments, after the others' totals
__global__ void __launch_bounds__(256) k_ul_starts(UlArgs A) {
    __shared__ double s_tot[8][32];
    const int nsl = (A.d + 31) >> 5, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int64_t items = (int64_t)*A.n_large * nsl;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int64_t j = (int64_t)(A.order[it / nsl] & 0xFFFFFFFFull);
        const int t = (int)(it % nsl) * 32 + lane;
        const int64_t ns = ((int64_t)A.cnt[j] + UL_M - 1) / UL_M;
        const int64_t b0 = ns * w / 8, b1 = t < A.d ? ns * (w + 1) / 8 : b0;
        double *p = A.start + A.seg_off[j] * A.d + t;
        double run = 0.0;
        for (int pass = 0; pass < 2; pass++) {
            for (int64_t s0 = b0; s0 < b1; s0 += 16) {
                double v[16];
#pragma unroll
                for (int u = 0; u < 16; u++) v[u] = s0 + u < b1 ? p[(s0 + u) * A.d] : 0.0;
#pragma unroll
                for (int u = 0; u < 16; u++) {
                    if (pass && s0 + u < b1) p[(s0 + u) * A.d] = run;
                    run += v[u];
                }
            }
            if (pass == 0) {
                s_tot[w][lane] = run;
                __syncthreads();
                run = 0.0;
                for (int q = 0; q < w; q++) run += s_tot[q][lane];
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(256) k_ul_deltas(UlArgs A) {
    const int nsl = (A.d + 31) >> 5;
    const int64_t items = *A.n_seg * nsl, nw = ((int64_t)gridDim.x * blockDim.x) >> 5;
    for (int64_t it = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; it < items; it += nw) {
        const UlItem q = ul_item(A, it, nsl);
        const int64_t at = q.seg * A.d + q.t;
        const double s = q.act ? A.start[at] : 0.0;
        const int E = (int)(((uint64_t)__double_as_longlong(s) >> 52) & 0x7FF);
        bool ok = E > 64 && E < 0x7FE - 64;
        int64_t D0 = 0, D1 = 0, mn = 0, mx = 0;
        ul_rows(A, q, [&](float v) {
            // v / q = m 2^sh, m a 24-bit integer
            const uint32_t b = __float_as_uint(v);
            const int e = (int)((b >> 23) & 0xFFu);
            const int32_t ma = (int32_t)((b & 0x7FFFFFu) | ((uint32_t)min(e, 1) << 23));
            const int32_t m = (b >> 31) ? -ma : ma;
            const int sh = max(e, 1) + 925 - E;
            ok = ok && sh <= 28 && e != 0xFF;  // 128 values of at most 2^52 units each: no overflow
            int64_t r0, r1;
            if (sh >= 0) {
                r0 = r1 = (int64_t)((uint64_t)(int64_t)m << min(sh, 28));
            } else if (sh < -25) {
                r0 = r1 = 0;  // below half a unit
            } else {
                const int32_t F = m >> -sh, rem = m & ((1 << -sh) - 1), half = 1 << (-sh - 1);
                r0 = r1 = F + (rem > half);
                if (rem == half) {  // a tie: to the even one of S + F, S + F + 1
                    r0 = F + ((D0 + F) & 1);
                    r1 = F + ((1 + D1 + F) & 1);
                }
            }
            D0 += r0;
            D1 += r1;
            mn = min(mn, min(D0, D1));
            mx = max(mx, max(D0, D1));
        });
        if (q.act) ul_pack(A.rec + at, A.segs * A.d, D0, D1, mn, mx, E, ok);
    }
}

__global__ void __launch_bounds__(32) k_ul_chain(UlArgs A) {
    const int nsl = (A.d + 31) >> 5, lane = threadIdx.x;
    const int64_t items = (int64_t)*A.n_large * nsl;
    constexpr int64_t LO = (1ll << 52) + 1, HI = (1ll << 53) - 1;
    for (int64_t it = blockIdx.x; it < items; it += gridDim.x) {
        const int64_t j = (int64_t)(A.order[it / nsl] & 0xFFFFFFFFull);
        const int t = (int)(it % nsl) * 32 + lane;
        const bool act = t < A.d;
        const int64_t cj = (int64_t)A.cnt[j], ns = (cj + UL_M - 1) / UL_M;
        const int32_t *mid = A.ids + A.off[j];
        const float *xs = A.x + (act ? t : 0);
        const int64_t a0 = A.seg_off[j] * A.d + (act ? t : 0);
        double s = 0.0;
        // UL_U segments' words at a time, the next ones on the way meanwhile
        constexpr int UL_U = 4;
        const int64_t stride = A.segs * A.d;
        int64_t nw[UL_U][3];
        auto fetch = [&](int64_t g0) {
#pragma unroll
            for (int u = 0; u < UL_U; u++) {
                const int64_t *w = A.rec + a0 + min(g0 + u, ns - 1) * A.d;
                nw[u][0] = w[0];
                nw[u][1] = w[stride];
                nw[u][2] = w[2 * stride];
            }
        };
        fetch(0);
        for (int64_t g0 = 0; g0 < ns; g0 += UL_U) {
            int64_t cw[UL_U][3];
#pragma unroll
            for (int u = 0; u < UL_U; u++)
#pragma unroll
                for (int q = 0; q < 3; q++) cw[u][q] = nw[u][q];
            fetch(g0 + UL_U);
#pragma unroll
            for (int u = 0; u < UL_U; u++) {
                if (g0 + u >= ns) break;
                const int64_t D0 = cw[u][0] >> 2, D1 = D0 + (cw[u][0] & 3) - 1, mn = cw[u][1] >> 8, mx = cw[u][2] >> 8;
                const int ex = (int)(cw[u][1] & 0xFF) | (int)(cw[u][2] & 0xFF) << 8;  // 0x700 and more: not usable
                const uint64_t bits = (uint64_t)__double_as_longlong(s);
                const int E = (int)((bits >> 52) & 0x7FF);
                const int64_t a = (int64_t)((bits & ((1ull << 52) - 1)) | (1ull << 52));
                const bool neg = bits >> 63;
                const int64_t S = neg ? -a : a;
                const bool ok = !act || (ex == E && (neg ? S + mx <= -LO && S + mn >= -HI : S + mn >= LO && S + mx <= HI));
                const int64_t T = S + ((S & 1) ? D1 : D0);
                const uint64_t b = (uint64_t)(T < 0 ? -T : T);
                const double moved = __longlong_as_double(
                    (long long)((bits & (1ull << 63)) | ((uint64_t)E << 52) | (b & ((1ull << 52) - 1))));
                double walked = s;
                if (!__all_sync(0xffffffffu, ok)) {
                    const int64_t m0 = (g0 + u) * UL_M;
                    float w[UC_B];  // the next chunk's rows, requested before this one's sums
                    auto rows = [&](int64_t p) {
                        const int32_t id = p + lane < cj ? mid[p + lane] : 0;
#pragma unroll
                        for (int r = 0; r < UC_B; r++) {
                            const int32_t row = __shfl_sync(0xffffffffu, id, r);
                            w[r] = p + r < cj ? xs[(int64_t)row * A.ldx] : 0.f;
                        }
                    };
                    rows(m0);
                    for (int64_t p = m0; p < min(cj, m0 + UL_M); p += UC_B) {
                        const int ma = (int)min((int64_t)UC_B, cj - p);
                        float v[UC_B];
#pragma unroll
                        for (int r = 0; r < UC_B; r++) v[r] = w[r];
                        if (p + UC_B < min(cj, m0 + UL_M)) rows(p + UC_B);
                        walked = ma == UC_B ? chain_chunk<true>(walked, v, ma, act && !ok)
                                            : chain_chunk<false>(walked, v, ma, act && !ok);
                    }
                }
                s = ok ? moved : walked;
            }
        }
        if (act) A.c[j * A.d + t] = __ddiv_rn(s, (double)cj);
    }
}

// A second stream for work beside the caller's, for one call (some 30 us to make
// and give back, which a million rows outweigh; without one the work stays on the
// caller's).  fork: its work follows what st holds now; join: st's next work
// follows its own.  A Joined in the scope of the buffers joins before they are
// given back, also when the call ends early.
constexpr int64_t SIDE_MIN = 1 << 20;
struct SideStream {
    cudaStream_t st, s = nullptr;
    cudaEvent_t ev = nullptr;
    bool on = false, forked = false;
    explicit SideStream(cudaStream_t main) : st(main) {}
    void open() {
        on = cudaStreamCreateWithFlags(&s, cudaStreamNonBlocking) == cudaSuccess &&
             cudaEventCreateWithFlags(&ev, cudaEventDisableTiming) == cudaSuccess;
        if (!on) cudaGetLastError();
    }
    cudaError_t fork() {
        const cudaError_t e = cudaEventRecord(ev, st);
        if (e != cudaSuccess) return e;
        forked = true;
        return cudaStreamWaitEvent(s, ev, 0);
    }
    cudaError_t join() {
        if (!forked) return cudaSuccess;
        forked = false;
        const cudaError_t e = cudaEventRecord(ev, s);
        return e == cudaSuccess ? cudaStreamWaitEvent(st, ev, 0) : e;
    }
    ~SideStream() {
        if (ev) cudaEventDestroy(ev);
        if (s) cudaStreamDestroy(s);
    }
    SideStream(const SideStream &) = delete;
    SideStream &operator=(const SideStream &) = delete;
};
struct Joined {
    SideStream &side;
    ~Joined() { side.join(); }
};

geek_status refine_dense(geek_ctx *ctx, Scratch &scr, const float *x, int64_t ldx, int64_t n, int d, double *centres,
                         int64_t k, int passes, int precision, int32_t *labels, geek_assign_stats *stats,
                         cudaStream_t st) {
    // The rows' conversion serves every pass.  With many rows it runs beside the
    // first centre update, on a second stream.
    TcX xc;
    const bool tc = (precision == GEEK_PREC_BF16 || precision == GEEK_PREC_BF16X3) && d <= 128;
    Scratch xs(ctx, st);
    SideStream side(st);
    if (passes > 0 && k > 0 && n >= SIDE_MIN) side.open();
    if (passes > 0 && k > 0 && n > 0 && tc) GK_TRY(tc_x_alloc(ctx, xs, n, d, precision == GEEK_PREC_BF16X3, &xc));
    for (int pass = 0; pass < passes && n > 0 && k > 0; pass++) {
        Scratch ps(ctx, st);
        Joined joined{side};
        uint64_t *key;
        uint32_t *ids;
        unsigned long long *cnt;
        int64_t *off;
        int *bad;
        GK_TRY(ps.alloc(&key, n));
        GK_TRY(ps.alloc(&ids, n));
        GK_TRY(ps.alloc(&cnt, k));
        GK_TRY(ps.alloc(&off, k));
        GK_TRY(ps.alloc(&bad, 1));
        EvTimer tg(ctx, "refine.group", st);
        GK_CUDA(ctx, cudaMemsetAsync(cnt, 0, sizeof(unsigned long long) * k, st));
        GK_CUDA(ctx, cudaMemsetAsync(bad, 0, sizeof(int), st));
        GK_COUNT();
        k_label_keys<<<grid_for(n, 256, ctx->num_sms), 256, 0, st>>>(n, labels, k, key, ids, cnt, bad);
        GK_LAUNCH(ctx);
        GK_TRY(radix_sort_segments(ctx, ps, 1, n, &key, nullptr, &ids, bit_length_u64((uint64_t)k), st));
        GK_TRY(exclusive_scan_i64(ctx, ps, (const int64_t *)cnt, off, k, nullptr, st));
        uint64_t *order;
        int64_t *nseg, *seg_off, *seg_tot;
        unsigned long long *n_large;
        GK_TRY(ps.alloc(&order, k));
        GK_TRY(ps.alloc(&nseg, k));
        GK_TRY(ps.alloc(&seg_off, k));
        GK_TRY(ps.alloc(&seg_tot, 1));
        GK_TRY(ps.alloc(&n_large, 1));
        // the segments' arrays (at most so many), n d / 4 bytes; without room for them
        // every centre is one chain
        UlArgs U{x, ldx, d, k, off, cnt, (const int32_t *)ids, seg_off, seg_tot, nullptr, n_large};
        U.segs = n / UL_M + n / UL_MIN + 1;
        U.c = centres;
        bool cut = n > UL_MIN;  // else no centre is large
        if (cut) GK_TRY(ps.try_alloc(&U.start, (size_t)U.segs * d, &cut));
        if (cut) GK_TRY(ps.try_alloc(&U.rec, 3 * (size_t)U.segs * d, &cut));
        if (!cut) GK_CUDA(ctx, cudaMemsetAsync(n_large, 0, sizeof(unsigned long long), st));
        GK_COUNT();
        k_size_order<<<grid_for(k, 256, ctx->num_sms), 256, 0, st>>>(k, cnt, order, nseg);
        GK_LAUNCH(ctx);
        GK_TRY(radix_sort_segments(ctx, ps, 1, k, &order, nullptr, nullptr, 64, st));
        U.order = order;
        if (cut) {
            GK_COUNT();
            k_large<<<1, 256, 0, st>>>(k, std::min(k, n / UL_MIN), n, d, UC_P * ctx->num_sms, side.on, cnt, order, nseg,
                                       n_large);
            GK_LAUNCH(ctx);
            GK_TRY(exclusive_scan_i64(ctx, ps, nseg, seg_off, k, seg_tot, st));
        }
        tg.stop();
        unsigned long long *next;
        int *uc_err;
        GK_TRY(ps.alloc(&next, 1));
        GK_TRY(ps.alloc(&uc_err, 1));
        GK_CUDA(ctx, cudaMemsetAsync(next, 0, sizeof(unsigned long long), st));
        GK_CUDA(ctx, cudaMemsetAsync(uc_err, 0, sizeof(int), st));
        static bool uc_attr = false;
        if (!uc_attr) {
            GK_CUDA(ctx, cudaFuncSetAttribute(k_update_centres, cudaFuncAttributeMaxDynamicSharedMemorySize, UC_SMEM));
            uc_attr = true;
        }
        EvTimer tu(ctx, "kernel.update_centres", st);
        if (cut) {
            const int nsl = (d + 31) / 32;
            const int gs = grid_for(U.segs * nsl * 32, 256, ctx->num_sms);
            const int64_t most = (n / UL_MIN) * nsl;  // (large centre, slice) items, at most
            GK_COUNT();
            k_ul_sums<<<gs, 256, 0, st>>>(U);
            GK_COUNT();
            k_ul_starts<<<(unsigned)std::min<int64_t>(most, (int64_t)ctx->num_sms * 8), 256, 0, st>>>(U);
            GK_COUNT();
            k_ul_deltas<<<gs, 256, 0, st>>>(U);
            if (side.on) GK_CUDA(ctx, side.fork());  // with the chains that are not cut
            GK_COUNT();
            k_ul_chain<<<(unsigned)std::min<int64_t>(most, (int64_t)ctx->num_sms * 16), 32, 0, st>>>(U);
            GK_LAUNCH(ctx);
        }
        const cudaStream_t us = cut && side.on ? side.s : st;
        GK_COUNT();
        k_update_centres<<<(unsigned)std::min<int64_t>((k * ((d + 31) / 32) + UC_P - 1) / UC_P, (int64_t)ctx->num_sms),
                           UC_T, UC_SMEM, us>>>(x, ldx, d, k, off, cnt, (const int32_t *)ids, order, n_large, next,
                                                centres, uc_err);
        GK_LAUNCH(ctx);
        if (tc && pass == 0) GK_TRY(tc_x_convert(ctx, x, ldx, n, d, precision == GEEK_PREC_BF16X3, xc, us));
        GK_CUDA(ctx, side.join());
        tu.stop();
        int h_bad = 0, h_uc = 0;
        GK_CUDA(ctx, cudaMemcpyAsync(&h_bad, bad, sizeof h_bad, cudaMemcpyDeviceToHost, st));
        GK_CUDA(ctx, cudaMemcpyAsync(&h_uc, uc_err, sizeof h_uc, cudaMemcpyDeviceToHost, st));
        GK_TRY(sort_err_check(ctx, st));  // synchronises st
        if (h_bad) return set_error(ctx, GEEK_ERR_INVALID, "a label outside [-1, k)");
        if (h_uc) return set_error(ctx, (geek_status)h_uc, "centre update: a pipeline wait timed out");
        EvTimer ta(ctx, "refine.assign", st);
        // the statistics describe the last pass only
        GK_TRY(assign_dense_centres(ctx, ps, x, ldx, n, d, centres, k, precision, labels,
                                    pass + 1 == passes ? stats : nullptr, st, tc ? &xc : nullptr));
    }
    return GEEK_OK;
}

// After decide_flags: the candidates' pass ran to its end, and so did the sort of
// the flagged rows (its word is read, and cleared, in the same wait).
static geek_status decide_check(geek_ctx *ctx, const TcPlan &P, cudaStream_t st) {
    int h_sort = 0;
    GK_TRY(sort_err_fetch(ctx, &h_sort, st));
    const geek_status pass = tc_plan_check(ctx, P, st);  // synchronises
    const geek_status sort = sort_err_eval(ctx, &h_sort, st);
    return pass != GEEK_OK ? pass : sort;
}

geek_status assign_dense_centres(geek_ctx *ctx, Scratch &scr, const float *x, int64_t ldx, int64_t n, int d,
                                 const double *centres, int64_t k, int precision, int32_t *labels,
                                 geek_assign_stats *stats, cudaStream_t st, const TcX *xc) {
    if (stats) *stats = geek_assign_stats{0.0, 0.0, k, 0};
    if (n == 0) return GEEK_OK;
    if (k == 0) {
        GK_COUNT();
        k_fill_labels<<<grid_for(n, 256, ctx->num_sms), 256, 0, st>>>(labels, n, -1);
        GK_LAUNCH(ctx);
        return GEEK_OK;
    }
    if (d > AS_MAXD) return set_error(ctx, GEEK_ERR_UNSUPPORTED, "dense assignment supports d <= %d", AS_MAXD);
    if (precision != GEEK_PREC_FP32 && precision != GEEK_PREC_BF16 && precision != GEEK_PREC_BF16X3)
        return set_error(ctx, GEEK_ERR_INVALID, "bad precision");
    // the call's small words and tables share one allocation and one fill
    struct Words {
        unsigned long long n_flag;
        double stats[2];
        unsigned cmax_bits;
        OneTables one;
    } *w;
    float *c32, *cn;
    GK_TRY(scr.alloc(&w, 1));
    GK_TRY(scr.alloc(&c32, (size_t)k * (d + 1)));
    cn = c32 + (size_t)k * d;
    GK_CUDA(ctx, cudaMemsetAsync(w, 0, sizeof(Words), st));
    unsigned long long *n_flag = &w->n_flag;
    const RInst *ri = &w->one.r;
    const int64_t *roff = w->one.row_off;
    {
        const CInst hc{centres, c32, cn, &w->cmax_bits, d, 0};
        const OneTables one{RInst{x, ldx, d, c32, cn, centres, k, &w->cmax_bits, labels, 0}, {0, n}};
        GK_COUNT();
        const CentreWarp cw = centre_warp(ctx, k);
        k_centre_prep_one<<<grid_for(ceil_div(k, cw.centres()) * 32, 128, ctx->num_sms), 128, 0, st>>>(hc, k, cw, one,
                                                                                                      &w->one);
        GK_LAUNCH(ctx);
    }
    int32_t *flag_rows;
    float *flag_m;  // the fast pass's smallest value per flagged row
    GK_TRY(scr.alloc(&flag_rows, n));
    GK_TRY(scr.alloc(&flag_m, n));
    TcPlan plan;
    struct Free {
        TcPlan *p;
        ~Free() { tc_plan_free(p); }
    } plan_free{&plan};
    if (precision == GEEK_PREC_BF16 || precision == GEEK_PREC_BF16X3) {
        plan.x_done = xc;
        GK_TRY(assign_tc_bf16(ctx, scr, x, ldx, n, d, centres, k, precision == GEEK_PREC_BF16X3, labels, flag_rows,
                              flag_m, n_flag, &plan, st));
    } else {
        const bool narrow = fp32_narrow(ctx, n, d);
        const size_t smem = fp32_smem(d, narrow);
        auto *const kernel = narrow ? k_assign_fp32<false, 16, 2> : k_assign_fp32<false, 32, 3>;
        GK_CUDA(ctx, cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                          (int)fp32_smem(AS_MAXD, false)));
        EvTimer tk(ctx, "kernel.assign_fp32", st);
        tk.work = 2.0 * (double)n * (double)k * (double)d;
        FArgs A{x, ldx, n, d, c32, cn, k, &w->cmax_bits, labels, flag_rows, flag_m, n_flag, ceil_div(n, AS_TR)};
        GK_COUNT();
        kernel<<<(unsigned)A.ntiles, 256, smem, st>>>(A, GatherUnits{});
        GK_LAUNCH(ctx);
    }
    unsigned long long h_flag = 0, h_fp64 = 0;
    DecideBufs db;
    if (precision == GEEK_PREC_FP32) {
        // the FP32 pass already applied the FP32 window: straight to FP64.  The
        // kernel reads the row count itself, so that the host need not wait
        // for it (with none it ends at once)
        EvTimer tk(ctx, "kernel.assign_recheck", st);
        GK_COUNT();
        k_assign_recheck<<<(unsigned)std::min<int64_t>(ceil_div(n, 8), (int64_t)ctx->num_sms * 8), 256, 0, st>>>(
            ri, roff, 1, flag_rows, flag_m, n_flag);
        GK_LAUNCH(ctx);
    } else {
        GK_CUDA(ctx, cudaMemcpyAsync(&h_flag, n_flag, sizeof h_flag, cudaMemcpyDeviceToHost, st));
        GK_TRY(tc_plan_check(ctx, plan, st));  // synchronises
        if (h_flag) {
            GK_TRY(decide_bufs_alloc(ctx, &scr, 1, n, db));
            GK_TRY(tc_emit_alloc(ctx, &scr, &plan, (int64_t)h_flag, st));
            // the label order pays for its sort from some 10^5 rows on (all rows flagged,
            // 128 dimensions, k = 2,000, decision with and without: 50,000 rows 1.79 and
            // 1.76 ms, 100,000 2.18 and 2.24, 500,000 3.53 and 4.19; 32 dimensions 0.52 and
            // 0.50, 0.66 and 0.69, 1.46 and 1.84)
            const FlagOrder order{&scr, k, labels};
            GK_TRY(decide_flags(ctx, plan, ri, roff, 1, d, flag_rows, flag_m, n_flag, (int64_t)h_flag, db, st,
                                h_flag >= 100000 ? &order : nullptr));
            if (!stats) GK_TRY(decide_check(ctx, plan, st));
        }
    }
    if (stats) {
        const int nb = grid_for(n, 256, ctx->num_sms);
        double *ps;
        float *pm;
        GK_TRY(scr.alloc(&ps, nb));
        GK_TRY(scr.alloc(&pm, nb));
        float *chi, *clo;
        GK_TRY(scr.alloc(&chi, (size_t)k * d));
        GK_TRY(scr.alloc(&clo, (size_t)k * d));
        GK_COUNT();
        k_centre_split<<<grid_for(k * d, 256, ctx->num_sms), 256, 0, st>>>(centres, k * d, chi, clo);
        GK_COUNT();
        k_assign_stats<<<nb, 256, 0, st>>>(x, ldx, n, d, chi, clo, k, labels, ps, pm);
        GK_COUNT();
        k_stats_final<<<1, 256, 0, st>>>(ps, pm, nb, w->stats);
        GK_LAUNCH(ctx);
        Words h;
        GK_CUDA(ctx, cudaMemcpyAsync(&h, w, offsetof(Words, cmax_bits), cudaMemcpyDeviceToHost, st));
        if (h_flag) {
            GK_CUDA(ctx, cudaMemcpyAsync(&h_fp64, db.n_flag2, sizeof h_fp64, cudaMemcpyDeviceToHost, st));
            GK_TRY(decide_check(ctx, plan, st));  // synchronises
        } else {
            GK_CUDA(ctx, cudaStreamSynchronize(st));
        }
        if (precision == GEEK_PREC_FP32) h_flag = h_fp64 = h.n_flag;
        stats->sse = h.stats[0];
        stats->radius_max = h.stats[1];
        stats->k = k;
        stats->n_recheck_rows = (int64_t)h_flag;
        stats->n_fp64_rows = (int64_t)h_fp64;
    }
    return GEEK_OK;
}

geek_status centroids_batch(geek_ctx *ctx, const CenInst *C, const int64_t *seed_inst_off, int count, int64_t ktot,
                            int dmax, const int64_t *soff, const int32_t *sids, cudaStream_t st) {
    if (ktot == 0) return GEEK_OK;
    GK_COUNT();
    k_centroids_batch<<<grid_for(ktot * dmax, 256, ctx->num_sms), 256, 0, st>>>(C, seed_inst_off, count, ktot, dmax,
                                                                              soff, sids);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

geek_status centre_prep_batch(geek_ctx *ctx, const CInst *C, const int64_t *k_off, int count, int64_t ktot,
                              cudaStream_t st) {
    if (ktot == 0) return GEEK_OK;
    GK_COUNT();
    const CentreWarp cw = centre_warp(ctx, ktot);
    k_centre_prep<<<grid_for(ceil_div(ktot, cw.centres()) * 32, 128, ctx->num_sms), 128, 0, st>>>(C, k_off, count, ktot, cw);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}


geek_status centre_split(geek_ctx *ctx, const double *c64, int64_t total, float *chi, float *clo, cudaStream_t st) {
    if (total == 0) return GEEK_OK;
    GK_COUNT();
    k_centre_split<<<grid_for(total, 256, ctx->num_sms), 256, 0, st>>>(c64, total, chi, clo);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

geek_status stats_batch(geek_ctx *ctx, const SInst *S, const int2 *units, int64_t nunits, const int64_t *unit_off,
                        int count, double *part_sum, float *part_max, double *sse, double *rmax, cudaStream_t st) {
    if (nunits > 0) {
        GK_COUNT();
        k_assign_stats_batch<<<(int)std::min<int64_t>(nunits, (int64_t)ctx->num_sms * 16), 256, 0, st>>>(
            S, units, nunits, part_sum, part_max);
    }
    GK_COUNT();
    k_stats_final_batch<<<(count + 127) / 128, 128, 0, st>>>(part_sum, part_max, unit_off, count, sse, rmax);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

geek_status fill_labels(geek_ctx *ctx, int32_t *labels, int64_t n, int32_t v, cudaStream_t st) {
    if (n == 0) return GEEK_OK;
    GK_COUNT();
    k_fill_labels<<<grid_for(n, 256, ctx->num_sms), 256, 0, st>>>(labels, n, v);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

geek_status decide_bufs_alloc(geek_ctx *ctx, Scratch *scr, int count, int64_t n_total, DecideBufs &B) {
    const int64_t nu = ceil_div(n_total, AS_TR) + count;
    auto al = [&](auto **p, size_t c) -> geek_status {
        if (scr) return scr->alloc(p, c);
        void *q = nullptr;
        if (cudaMalloc(&q, std::max<size_t>(c * sizeof(**p), 16)) != cudaSuccess) {
            cudaGetLastError();
            return set_error(ctx, GEEK_ERR_NOMEM, "decision buffers");
        }
        B.owned.push_back(q);
        *p = (std::remove_reference_t<decltype(*p)>)q;
        return GEEK_OK;
    };
    GK_TRY(al(&B.cnt, count));
    GK_TRY(al(&B.cursor, count));
    GK_TRY(al(&B.unit_inst, nu));
    GK_TRY(al(&B.unit_start, nu));
    GK_TRY(al(&B.unit_cnt, nu));
    GK_TRY(al(&B.n_units, 1));
    GK_TRY(al(&B.seg_off, count + 1));
    GK_TRY(al(&B.unit_off, count + 1));
    GK_TRY(al(&B.left, std::max<int64_t>(n_total, 1)));
    GK_TRY(al(&B.n_left, 1));
    GK_TRY(al(&B.grows, std::max<int64_t>(n_total, 1)));
    GK_TRY(al(&B.flags2, std::max<int64_t>(n_total, 1)));
    GK_TRY(al(&B.flags2_m, std::max<int64_t>(n_total, 1)));
    GK_TRY(al(&B.mrow, std::max<int64_t>(n_total, 1)));
    GK_TRY(al(&B.n_flag2, 1));
    return GEEK_OK;
}

void decide_bufs_free(DecideBufs &B) {
    for (void *p : B.owned) cudaFree(p);
    B.owned.clear();
}

// one instance: the list is the group
__global__ void k_one_group(const int32_t *__restrict__ flags, const unsigned long long *__restrict__ n_flag,
                            int64_t *__restrict__ seg_off, int64_t *__restrict__ unit_off, int *__restrict__ n_units,
                            int32_t *__restrict__ grows) {
    const int64_t nf = (int64_t)*n_flag;
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nf; q += (int64_t)gridDim.x * blockDim.x)
        grows[q] = flags[q];
    if (blockIdx.x == 0 && threadIdx.x == 0) {
        const int64_t nu = (nf + AS_TR - 1) / AS_TR;
        seg_off[0] = unit_off[0] = 0;
        seg_off[1] = nf;
        unit_off[1] = nu;
        *n_units = (int)nu;
    }
}

// the listed rows grouped by instance in units of 128 (B.grows, B.unit_*); one
// instance's rows keep the list's order
static geek_status group_flags(geek_ctx *ctx, const int64_t *row_off, int count, const int32_t *flags,
                               const unsigned long long *n_flag, const DecideBufs &B, cudaStream_t st) {
    const int g = ctx->num_sms * 4;
    GK_COUNT();
    if (count == 1) {
        k_one_group<<<g, 256, 0, st>>>(flags, n_flag, B.seg_off, B.unit_off, B.n_units, B.grows);
    } else {
        GK_CUDA(ctx, cudaMemsetAsync(B.cnt, 0, sizeof(int) * count, st));
        k_flag_count<<<g, 256, 0, st>>>(flags, n_flag, row_off, count, B.cnt);
        GK_COUNT();
        k_flag_units<<<1, 1024, 0, st>>>(B.cnt, count, B.cursor, B.seg_off, B.unit_off, B.n_units);
        GK_COUNT();
        k_flag_scatter<<<g, 256, 0, st>>>(flags, n_flag, row_off, count, B.cursor, B.grows);
    }
    GK_COUNT();
    k_fill_units<<<g, 256, 0, st>>>(count, B.seg_off, B.unit_off, B.unit_inst, B.unit_start, B.unit_cnt);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

// (label, row) words of the flagged rows, and the rows of the sorted words
__global__ void k_flag_words(int64_t nf, const int32_t *__restrict__ flags, const int32_t *__restrict__ labels,
                             uint64_t *__restrict__ words) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nf; q += (int64_t)gridDim.x * blockDim.x) {
        const int32_t r = flags[q];
        words[q] = ((uint64_t)(uint32_t)max(labels[r], 0) << 32) | (uint32_t)r;
    }
}
__global__ void k_word_rows(int64_t nf, const uint64_t *__restrict__ words, int32_t *__restrict__ rows) {
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < nf; q += (int64_t)gridDim.x * blockDim.x)
        rows[q] = (int32_t)(uint32_t)words[q];
}

// One data set's nf flagged rows in the order of the label the fast pass gave
// them: neighbours then have the same candidates, whose centres the decision
// reads from L1 instead of L2 (Alg. 1 pipeline, 4.7M rows of 35 candidates:
// the decision takes 11 ms, 18 ms in the order of the flags).
static geek_status order_flags(geek_ctx *ctx, Scratch &scr, int64_t nf, int64_t k, const int32_t *labels,
                               int32_t *flags, cudaStream_t st) {
    uint64_t *words;
    GK_TRY(scr.alloc(&words, nf));
    GK_COUNT();
    k_flag_words<<<grid_for(nf, 256, ctx->num_sms), 256, 0, st>>>(nf, flags, labels, words);
    GK_LAUNCH(ctx);
    GK_TRY(radix_sort_segments(ctx, scr, 1, nf, &words, nullptr, nullptr, 32 + bit_length_u64((uint64_t)k), st, 32));
    GK_COUNT();
    k_word_rows<<<grid_for(nf, 256, ctx->num_sms), 256, 0, st>>>(nf, words, flags);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

// Decides the flagged rows of a tensor-core pass exactly (flags: global rows;
// flag_m: their smallest fast values).  Nearly all of them among their
// candidates, by direct FP32 distances (tc_decide_candidates); the rest (near
// duplicates of one centre, values that are not finite) by a tiled FP32 scan of
// every centre (narrow FP32 window), then the FP64 reference for the rows still
// uncertain.  max_rows: at most so many flagged rows.  No host synchronisation
// and no allocation, except with `order` (one data set, exactly max_rows flagged
// rows): flags is then put into the order of the labels first.
// Alg. 1 pipeline at 10M x 128, k = 1,751, split-BF16: 4.7M flagged rows of 35
// candidates each take 19 ms; the two scans over every centre took 162.
geek_status decide_flags(geek_ctx *ctx, const TcPlan &P, const RInst *R, const int64_t *row_off, int count, int dmax,
                         int32_t *flags, const float *flag_m, const unsigned long long *n_flag, int64_t max_rows,
                         const DecideBufs &B, cudaStream_t st, const FlagOrder *order) {
    EvTimer tk(ctx, "kernel.assign_recheck", st);
    const int g = ctx->num_sms * 4;
    const FlagUnits F{B.grows, B.unit_inst, B.unit_start, B.unit_cnt, B.n_units};
    GK_CUDA(ctx, cudaMemsetAsync(B.n_flag2, 0, sizeof(unsigned long long), st));
    GK_CUDA(ctx, cudaMemsetAsync(B.n_left, 0, sizeof(unsigned long long), st));
    GK_COUNT();
    k_scatter_m<<<g, 256, 0, st>>>(flags, flag_m, n_flag, B.mrow);
    if (order) GK_TRY(order_flags(ctx, *order->scr, max_rows, order->k, order->labels, flags, st));
    GK_TRY(group_flags(ctx, row_off, count, flags, n_flag, B, st));
    GK_TRY(tc_decide_candidates(ctx, P, R, F, B.mrow, max_rows, order != nullptr, B.left, B.n_left, st));
    GK_TRY(group_flags(ctx, row_off, count, B.left, B.n_left, B, st));
    const size_t smem = (size_t)dmax * AS_TR * sizeof(float) + (size_t)AS_KC * AS_TC * sizeof(float);
    auto *const scan = k_assign_fp32<true, 32, 3>;  // d <= 128
    GK_CUDA(ctx, cudaFuncSetAttribute(scan, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)fp32_smem(AS_MAXD, false)));
    FArgs A{};
    A.flag_rows = B.flags2;
    A.flag_m = B.flags2_m;
    A.n_flag = B.n_flag2;
    const GatherUnits U{R, F};
    EvTimer t32(ctx, "kernel.assign_refine32", st);
    GK_COUNT();
    scan<<<ctx->num_sms * 2, 256, fp32_smem(dmax, false), st>>>(A, U);
    GK_LAUNCH(ctx);
    t32.stop();
    // the rows still uncertain, grouped by instance again, go to the tiled
    // FP64 decision with their smallest FP32 value
    const size_t mx = (size_t)AS_MAXD * AS_TR * sizeof(float) + (size_t)AS_KC * AS_TC * sizeof(float) + DQ_BYTES;
    GK_CUDA(ctx, cudaFuncSetAttribute(k_assign_decide64, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)mx));
    GK_COUNT();
    k_scatter_m<<<g, 256, 0, st>>>(B.flags2, B.flags2_m, B.n_flag2, B.mrow);
    GK_TRY(group_flags(ctx, row_off, count, B.flags2, B.n_flag2, B, st));
    EvTimer t64(ctx, "kernel.assign_decide64", st);
    GK_COUNT();
    k_assign_decide64<<<ctx->num_sms * 2, 256, smem + DQ_BYTES, st>>>(U, B.mrow);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}

// radius[j] = sqrt(max over objects labelled j of their distance to centre
// j), 0 for a centre nobody is nearest to; labels outside [0, k) are skipped.
geek_status cluster_radius(geek_ctx *ctx, Scratch &scr, const float *x, int64_t ldx, int64_t n, int d,
                           const double *centres, int64_t k, const int32_t *labels, double *radius, cudaStream_t st) {
    if (k == 0) return GEEK_OK;
    float *chi, *clo;
    unsigned *rmax;
    GK_TRY(scr.alloc(&chi, (size_t)k * d));
    GK_TRY(scr.alloc(&clo, (size_t)k * d));
    GK_TRY(scr.alloc(&rmax, k));
    GK_CUDA(ctx, cudaMemsetAsync(rmax, 0, sizeof(unsigned) * k, st));
    GK_COUNT();
    k_centre_split<<<grid_for(k * d, 256, ctx->num_sms), 256, 0, st>>>(centres, k * d, chi, clo);
    if (n > 0) {
        GK_COUNT();
        k_cluster_rmax<<<grid_for(n * 32, 256, ctx->num_sms), 256, 0, st>>>(x, ldx, n, d, chi, clo, k, labels, rmax);
    }
    GK_COUNT();
    k_cluster_sqrt<<<grid_for(k, 256, ctx->num_sms), 256, 0, st>>>(k, rmax, radius);
    GK_LAUNCH(ctx);
    return GEEK_OK;
}
