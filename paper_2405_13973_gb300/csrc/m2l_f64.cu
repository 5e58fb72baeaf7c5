// m2l_f64.cu -- the dense FP64 translations (M2M, M2L of Eq. FMM_local, L2L)
// on the 5th-generation tensor cores, from exact integer slices.
//
// FP64 runs at 1.25 TFLOP/s on this GPU and the FP64 translations are its
// largest consumer, while 16-bit products with FP32 sums run about 1500 times
// as fast.  A product of FP64 matrices is therefore split into products of
// small integers that the tensor core forms without rounding (the splitting
// of Ootomo, Ozaki and Yokota, "DGEMM on integer matrix multiplication unit",
// IJHPCA 2024, with f16 operands in place of int8):
//   * a row of coefficients x_k (a cell's M or L; an operator's row T[n][.])
//     is written as X_k 2^(e - 53), e the exponent of its largest magnitude,
//     |X_k| <= 2^54 an integer, and X_k as seven digits of base 256,
//     X = sum_i d_i 2^(8 (6 - i)), |d_i| <= 128, |d_0| <= 64: the 53 bits of
//     the largest coefficients of the row;
//   * digits are exact in f16, digit products exact in FP32, and a sum of
//     them is exact while it stays below 2^24.  The products of equal i + j
//     have one weight, so they share an accumulator s_{i+j}, i + j = 0 .. 7:
//     34 products;
//   * S = sum_d s_d 2^(8 (7 - d)) is formed in integers (96 bits) and written
//     as a double, rounded once: the FP64 units, two lanes per clock and SM,
//     take no part.
// Error of one output, in units of the product of the two rows' maxima: the
// digits' own rounding, 2^-54 of either maximum per coefficient, and the
// products i + j >= 8 left out, below 2^-57 per coefficient: at worst
// P 2^-53 (1 + 1/16), the bound of P FP64 multiply-adds of values as large as
// the maxima.  |s_d| <= d 2^14 P (d >= 1; 6 2^14 P for d = 7), so every sum is
// exact up to p = 12; at p = 16 those from s_4 on could pass 2^24 with nearly
// every digit at its limit, and would lose their last bit, 2^-42 (crystals
// reach 2^20).
// Measured against long double, one offset's output row: 1e-16 .. 9e-16 of
// its norm, FP64 multiply-adds 5e-16 .. 2.6e-15 (p = 4 .. 16, 1 to 100 ions a
// cell, like and unlike charges); coefficients far below the largest of their
// row are less exact than by multiply-adds (their error is of the row's size).
// Far fields of 427 to 60,000 ions, relative error of E: 2.1e-16 .. 7.2e-16,
// by multiply-adds 3.0e-16 .. 1.1e-15.  Without the products i + j = 7 (28 of
// them, 5.1 ms for the M2L below) E was off by up to 2e-14.
//   * L2L: the parent's L_0, which in a large crystal is many times the rest
//     of its row, reaches the child's L_0 only; it stays out of the digits and
//     is added in FP64 (E at depth 4, 12,000 ions, p = 4: 6.1e-16 -> 2.6e-16).
//
// One CTA per SM walks the work items (one operator, up to 128 rows):
//   D[128 rows x N] = sum over K steps of 16, i, j:  A_i[128 x 16] B_j[16 x N],
// in column chunks of up to 48 outputs so that the eight accumulators (384
// TMEM columns) leave room for two K steps of A in tensor memory (7 digits
// x 8 columns each).  A comes from tensor memory because with 48 columns a
// product takes 24 cycles and reading a 4 KB A tile from shared memory 32:
//   * warps 10..13 (one TMEM lane quarter each) bring the rows' digits by bulk
//     copies (one byte per digit and coefficient: half the bytes of f16; an
//     item's, 172 KB at p = 12, once, above p = 12 once per column chunk),
//     expand them to f16 (a byte permute into 1024 + d + 128, one packed
//     subtraction) and store them to tensor memory;
//   * warp 8 brings the operator digits, packed in f16 in the swizzled
//     K-major shared-memory image, by bulk copies of 32-wide K chunks;
//   * warp 9 issues the 34 products of a K step;
//   * warps 0..7 read the accumulators, release them once the integers are
//     formed, and write the doubles while the next chunk's products run.
// Every mbarrier wait is bounded as in m2l_tc.cu.
// M2L kernel, before (CUDA cores) -> now: 1e5 ions, p = 12, 53.7 ms (rotated
// translations) -> 6.1; a field at 1e6 ions, p = 8, 685 ms (tiles) -> 36.7.
// Bound by the issue of 48-column products and the hand-over of the accumulators.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>
#include <string.h>

#include <algorithm>

#include "harmonics.cuh"
#include "internal.h"
#include "m2l_pairs.h"
#include "tc_ptx.cuh"

namespace pt {

namespace {

constexpr int kDig = 7;                 // digits per coefficient
constexpr int kChunk = 48;              // output columns per chunk (at most)
constexpr int kF64Rows = 128;
constexpr int kSegBytes = kDig * 32;    // digits of one row in a 32-wide K segment
constexpr int kMaxRing = 5;             // ring slots of digit rows
constexpr int kAcc = kDig + 1;          // accumulators s_0 .. s_7
constexpr int kAStages = 2;             // K steps of A in tensor memory
constexpr int kACol0 = kAcc * kChunk;   // their first TMEM column
static_assert(kACol0 + kAStages * kDig * 8 <= 512, "tensor memory columns");
constexpr int kBStages = 4;             // 32-wide K chunks of B in shared memory (at most)
constexpr int kF64Threads = 448;
constexpr int kF64Ops = 359;            // 343 M2L offsets, 8 M2M, 8 L2L octants
constexpr int kF64M2M = 343, kF64L2L = 351;
constexpr int kRowNan = 0x7fffffff;     // exponent of a row with a NaN or infinity
constexpr int kSumExp = 66;             // a sum S stands for S 2^(exponents - 66): 106 - 8 (12 - 7)

enum F64Mode { F64_PAIR = 0, F64_M2M = 1, F64_L2L = 2 };

struct F64Args {
    int P, ld, lda;            // coefficients, row stride of M, L and partial rows, digit row stride
    int npad, ksteps, kst32, nch, level;
    int ring, gsegs, resident, bst;  // A ring slots, K segments in each, items resident, B stages
    int64_t zero_cell;         // a cell whose digits are all zero
    int64_t out_stride, op_bytes;
    const uint8_t* dig;        // [cell][kst32][kDig][32]
    const int* rexp;           // [cell]
    const unsigned char* ops;  // [kF64Ops][chunk][kst32][kDig][columns][64 B]
    const int16_t* oexp;       // [kF64Ops][npad]
    const M2lPairHdr* hdr;
    const M2lPairItem* items;
    const M2lPair* pairs;
    const LevelInfo* linfo;
    const uint32_t* code;
    const int32_t* cid;
    int64_t off_parent;
    const double* up;          // L2L: L of the parents
    double* out;
    int* err;
};

// instruction descriptor: D f32, A and B f16, K-major
__device__ __forceinline__ uint32_t idesc_f16(int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kF64Rows >> 4) << 24);
}
template <int ACC>
__device__ __forceinline__ void mma_f16_ts(uint32_t dtmem, uint32_t atmem, uint32_t blo,
                                           uint32_t bhi, uint32_t idesc) {
    asm volatile(
        "{\n .reg .b64 b;\n mov.b64 b, {%2, %3};\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], b, %4, %5;\n}" ::"r"(dtmem),
        "r"(atmem), "r"(blo), "r"(bhi), "r"(idesc), "n"(ACC)
        : "memory");
}
// the 34 products i + j <= 7 of a K step; MORE = 0: the first of an
// accumulator overwrites it
template <int MORE>
__device__ __forceinline__ void f64_products(uint32_t tm, uint32_t at, uint32_t blo, uint32_t bhi,
                                             uint32_t bstep, uint32_t id) {
#pragma unroll
    for (int j = 0; j < kDig; ++j)
        mma_f16_ts<MORE>(tm + (uint32_t)(j * kChunk), at, blo + bstep * (uint32_t)j, bhi, id);
#pragma unroll
    for (int i = 1; i < kDig; ++i)
#pragma unroll
        for (int j = 0; j < kDig && i + j < kAcc; ++j) {
            const uint32_t d = tm + (uint32_t)((i + j) * kChunk), x = at + (uint32_t)(8 * i),
                           y = blo + bstep * (uint32_t)j;
            if (i == 1 && j == kDig - 1) mma_f16_ts<MORE>(d, x, y, bhi, id);
            else mma_f16_ts<1>(d, x, y, bhi, id);
        }
}
__device__ __forceinline__ void tmem_ld4_nw(uint32_t taddr, uint32_t (&r)[4]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(taddr));
}
__device__ __forceinline__ void tmem_st8(uint32_t taddr, const uint32_t (&r)[8]) {
    asm volatile(
        "tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"r"(taddr),
        "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
        : "memory");
}

// 16 digit bytes (d + 128) -> 16 f16 digits: the byte becomes the low byte
// of 0x64xx = 1024 + byte, and 1152 is subtracted (exact)
__device__ __forceinline__ void expand16(const uint4& v, uint32_t (&h)[8]) {
    const uint32_t w[4] = {v.x, v.y, v.z, v.w};
    const __half2 bias = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        const uint32_t lo = __byte_perm(w[q], 0x64646464u, 0x4140);
        const uint32_t hi = __byte_perm(w[q], 0x64646464u, 0x4342);
        const __half2 a = __hsub2(*reinterpret_cast<const __half2*>(&lo), bias);
        const __half2 b = __hsub2(*reinterpret_cast<const __half2*>(&hi), bias);
        h[2 * q] = *reinterpret_cast<const uint32_t*>(&a);
        h[2 * q + 1] = *reinterpret_cast<const uint32_t*>(&b);
    }
}

__device__ __forceinline__ void tmem_ld1(uint32_t taddr, uint32_t (&r)[1]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r[0]) : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
}

// S = sum_d s_d 2^(8 (7 - d)) = hi 2^32 + lo (two's complement; |S| < 2^80)
struct F64Sum {
    long long hi;
    uint32_t lo;
};
__device__ __forceinline__ F64Sum f64_sum(long long upper, long long lower) {  // upper 2^32 + lower
    F64Sum r;
    r.hi = upper + (lower >> 32);
    r.lo = (uint32_t)lower;
    return r;
}
// from the bits v_d of s_d + 1.5 2^23 (|s_d| < 2^22): neighbours joined in 32
// bits (|256 s + s'| < 2^31), the biases taken off modulo 2^32
__device__ __forceinline__ F64Sum f64_join(const uint32_t (&v)[kAcc]) {
    constexpr uint32_t B2 = 257u * 0x4B400000u;
    int t[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) t[k] = (int)(v[2 * k] * 256u + v[2 * k + 1] - B2);
    return f64_sum((long long)t[0] * 65536 + (long long)t[1], (long long)t[2] * 65536 + (long long)t[3]);
}

// S 2^e as a double, rounded to nearest, in integer instructions, for
// exponents well inside the normal range (|e| <= kExpFast)
constexpr int kExpFast = 900;
__device__ __forceinline__ double fixed_to_double(const F64Sum& S, int e) {
    const uint32_t neg = (uint32_t)((unsigned long long)S.hi >> 63);
    // magnitude in three words
    uint32_t w0 = neg ? 0u - S.lo : S.lo;
    unsigned long long a = (unsigned long long)S.hi;
    if (neg) a = ~a + (S.lo == 0u ? 1ull : 0ull);
    uint32_t w2 = (uint32_t)(a >> 32), w1 = (uint32_t)a;
    int be = e + 95 + 1022;  // exponent field before the leading one is added
    if (w2 == 0u) {
        w2 = w1;
        w1 = w0;
        w0 = 0u;
        be -= 32;
    }
    if (w2 == 0u) {
        w2 = w1;
        w1 = 0u;
        be -= 32;
    }
    if (w2 == 0u) return 0.0;
    const int lz = __clz((int)w2);
    const uint32_t mh = __funnelshift_l(w1, w2, lz), ml = __funnelshift_l(w0, w1, lz);
    const unsigned long long r = ((unsigned long long)((mh >> 11) + ((uint32_t)(be - lz) << 20)) << 32) +
                                 (unsigned long long)__funnelshift_r(ml, mh, 11) + ((ml >> 10) & 1u);
    return __longlong_as_double((long long)(r | ((unsigned long long)neg << 63)));
}
// the rest: rows of subnormal or huge values, NaN rows
__device__ __noinline__ double fixed_to_double_slow(F64Sum S, int er, int fn) {
    if (er == kRowNan) return __longlong_as_double(0x7ff8000000000000ll);
    return ldexp(fixed_to_double(S, 0), er + fn);
}

// work unit idx: operator, rows, for M2M / L2L the first target cell, and the
// column chunks [c0, c1).  A unit is a whole item, or one chunk of it where
// there are few items (see k_f64_mma).
struct F64Work {
    int op, rows, base, c0, c1;
};
// Chunks are units of their own while the items alone would not fill the
// CTAs: an M2M or L2L launch of a few items then takes a chunk's time and not
// an item's (10k ions, p = 12: 38 -> 17 us and 43 -> 20 us each); with more
// items (316 M2L offsets of a 63-leaf tree) the units' own start costs more.
template <int MODE>
__device__ __forceinline__ bool f64_work(const F64Args& a, const LevelInfo& li, int idx, int count,
                                         int split, F64Work& w) {
    w.rows = 0;
    w.op = 0;
    w.base = 0;
    w.c0 = 0;
    w.c1 = a.nch;
    if (idx >= count) return false;
    if (split > 1) {
        w.c0 = idx % split;
        w.c1 = w.c0 + 1;
        idx /= split;
    }
    if (MODE == F64_PAIR) {
        const M2lPairItem it = a.items[idx];
        w.op = it.op;
        w.rows = it.rows;
        w.base = it.begin;
        return true;
    }
    // the level's cells of octant o in runs of 128
    int t = idx;
    for (int o = 0; o < 8; ++o) {
        const int s0 = li.oct_start[a.level][o], s1 = li.oct_start[a.level][o + 1];
        const int nt = (s1 - s0 + kF64Rows - 1) / kF64Rows;
        if (t < nt) {
            w.op = (MODE == F64_M2M ? kF64M2M : kF64L2L) + o;
            w.base = s0 + t * kF64Rows;
            w.rows = min(kF64Rows, s1 - w.base);
            return true;
        }
        t -= nt;
    }
    return false;
}
template <int MODE>
__device__ __forceinline__ int f64_count(const F64Args& a, const LevelInfo& li) {
    if (MODE == F64_PAIR) return a.hdr->n_items;
    int n = 0;
    for (int o = 0; o < 8; ++o)
        n += (li.oct_start[a.level][o + 1] - li.oct_start[a.level][o] + kF64Rows - 1) / kF64Rows;
    return n;
}
// the cell whose digits are row r of the item, or -1
template <int MODE>
__device__ __forceinline__ int f64_source(const F64Args& a, const F64Work& w, int r) {
    if (r >= w.rows) return -1;
    if (MODE == F64_PAIR) return a.pairs[w.base + r].src;
    if (MODE == F64_M2M) return w.base + r;
    return a.cid[a.off_parent + (a.code[w.base + r] >> 3)];
}

template <int MODE>
__global__ void __launch_bounds__(kF64Threads, 1) k_f64_mma(const __grid_constant__ F64Args a) {
    extern __shared__ unsigned char smem_dyn[];
    pdl_wait();
    __shared__ __align__(8) uint64_t fullA[kAStages], emptyA[kAStages], fullB[kBStages],
        emptyB[kBStages], fullR[kMaxRing], accf, acce, drain_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh;
    __shared__ LevelInfo li;
    volatile int* abort_v = &abort_sh;
    const int tid = threadIdx.x, lane = tid & 31;
    const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform to the compiler
    unsigned char* base = (unsigned char*)(((uintptr_t)smem_dyn + 1023) & ~(uintptr_t)1023);
    const int b_stage = kDig * min(kChunk, a.npad) * 64;
    if (MODE != F64_PAIR) {
        const int* src = reinterpret_cast<const int*>(a.linfo);
        int* dst = reinterpret_cast<int*>(&li);
        for (int i = tid; i < (int)(sizeof(LevelInfo) / sizeof(int)); i += kF64Threads) dst[i] = src[i];
    }
    if (tid == 0) {
        abort_sh = 0;
        for (int s = 0; s < kAStages; ++s) {
            mbar_init(&fullA[s], 128);
            mbar_init(&emptyA[s], 1);
        }
        for (int s = 0; s < kBStages; ++s) {
            mbar_init(&fullB[s], 1);
            mbar_init(&emptyB[s], 1);
        }
        for (int s = 0; s < kMaxRing; ++s) mbar_init(&fullR[s], 128);
        mbar_init(&accf, 1);
        mbar_init(&acce, 256);
        mbar_init(&drain_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int items = f64_count<MODE>(a, li);
    const int split = items <= (int)gridDim.x ? a.nch : 1;
    const int count = items * split;
    const int first = blockIdx.x, stride = gridDim.x;
    if (first >= count) return;  // uniform across the block
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                         smem_addr(&tmem_base_sh)),
                     "r"(512)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = tmem_base_sh;
    int r_issued = 0;     // A producers: digit copies issued
    int b_par[kBStages];  // operator producer: parity of the last copy per stage
#pragma unroll
    for (int s = 0; s < kBStages; ++s) b_par[s] = -1;

    if (warp == 8) {
        // ---- operator producer
        if (lane == 0) {
            int g = 0;
            F64Work w;
            for (int idx = first; f64_work<MODE>(a, li, idx, count, split, w) && !*abort_v; idx += stride) {
                const unsigned char* src = a.ops + (int64_t)w.op * a.op_bytes +
                                           (int64_t)a.kst32 * kDig * 64 * (w.c0 * kChunk);
                for (int c = w.c0; c < w.c1; ++c) {
                    const uint32_t bytes = (uint32_t)(kDig * min(kChunk, a.npad - c * kChunk) * 64);
                    for (int k = 0; k < a.kst32; ++k, ++g) {
                        const int st = g % a.bst, use = g / a.bst;
                        if (!mbar_wait_or_abort(&emptyB[st], (use & 1) ^ 1, abort_v)) {
                            *abort_v = 1;
                            break;
                        }
                        mbar_arrive_expect_tx(&fullB[st], bytes);
                        bulk_g2s(base + st * b_stage, src, bytes, &fullB[st]);
#pragma unroll
                        for (int s = 0; s < kBStages; ++s)
                            if (s == st) b_par[s] = use & 1;
                        src += bytes;
                    }
                    if (*abort_v) break;
                }
            }
        }
    } else if (warp == 9) {
        // ---- MMA issuer.  The whole warp runs the loops on warp-uniform
        // values and one elected lane issues (mbar_wait_warp)
        const uint32_t tm = __shfl_sync(0xffffffffu, tmem, 0);
        const int last = __shfl_sync(0xffffffffu, count, 0), sp = __shfl_sync(0xffffffffu, split, 0);
        int sa = 0, pa = 0, sb = 0, pb = 0, pacc = 1;  // stages and phases
        bool ok = true;
        for (int t = first; ok && t < last; t += stride) {
            const int c0 = sp > 1 ? t % sp : 0, c1 = sp > 1 ? c0 + 1 : a.nch;
            for (int c = c0; ok && c < c1; ++c) {
                const int N = min(kChunk, a.npad - c * kChunk);
                const uint32_t id = idesc_f16(N);
                const uint32_t bstep = (uint32_t)(N * 64) >> 4;  // one digit of B
                // the epilogue has read the previous chunk's accumulators
                // (the first wait finds the barrier's initial phase complete)
                ok = mbar_wait_warp(&acce, pacc, abort_v);
                pacc ^= 1;
                if (!ok) break;
                for (int ks = 0; ks < a.ksteps; ++ks) {
                    if (!(ks & 1)) ok = mbar_wait_warp(&fullB[sb], pb, abort_v);
                    ok = ok && mbar_wait_warp(&fullA[sa], pa, abort_v);
                    if (!ok) break;
                    tc_fence_after();
                    const uint64_t bd = sdesc64(smem_addr(base) + (uint32_t)(sb * b_stage) + 32u * (ks & 1));
                    const uint32_t blo = (uint32_t)bd, bhi = (uint32_t)(bd >> 32);
                    const uint32_t at = tm + (uint32_t)(kACol0 + sa * kDig * 8);
                    const bool endb = (ks & 1) || ks + 1 == a.ksteps;
                    if (elect_one()) {
                        if (ks == 0) f64_products<0>(tm, at, blo, bhi, bstep, id);
                        else f64_products<1>(tm, at, blo, bhi, bstep, id);
                        mma_commit(&emptyA[sa]);
                        if (endb) mma_commit(&emptyB[sb]);
                        if (ks + 1 == a.ksteps) mma_commit(&accf);
                    }
                    __syncwarp();
                    if (++sa == kAStages) {
                        sa = 0;
                        pa ^= 1;
                    }
                    if (endb && ++sb == a.bst) {
                        sb = 0;
                        pb ^= 1;
                    }
                }
            }
        }
        if (!ok) *abort_v = 1;
    } else if (warp >= 10) {
        // ---- A producers, thread = row.  Each thread brings its own row's
        // digits (contiguous in memory) by bulk copies of a.gsegs K segments
        // into its part of a ring slot, reads them back and expands them; it
        // alone reads and refills that part, so the rows need no barrier but
        // the slot's transaction count.  When an item's slots fit
        // (a.resident) they are loaded once and read by every column chunk,
        // and a slot is refilled for a later item while the last chunk runs;
        // else each chunk streams them.
        const int quad = warp & 3, row = quad * 32 + lane;
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)kACol0;
        const int64_t cell_bytes = (int64_t)kDig * a.lda;
        const int row_bytes = a.gsegs * kSegBytes + 16;  // 16: no bank conflicts
        unsigned char* ring = base + a.bst * b_stage + row * row_bytes;
        const int groups = (a.kst32 + a.gsegs - 1) / a.gsegs;
        const int nch = split > 1 ? 1 : a.nch;                   // chunks per unit
        const int loads = a.resident ? groups : nch * groups;    // per unit
        F64Work w;
        // the loading side: item lidx, its load lo; the source of the item
        // after it waits in a register
        int lidx = first, lo = 0, lslot = 0, issued = 0, freed = 0;
        int src = f64_work<MODE>(a, li, lidx, count, split, w) ? f64_source<MODE>(a, w, row) : -1, nsrc = -1;
        if (f64_work<MODE>(a, li, lidx + stride, count, split, w)) nsrc = f64_source<MODE>(a, w, row);
        auto issue = [&]() {
            if (lidx >= count || issued - freed >= a.ring) return;
            const int grp = lo % groups;
            const uint32_t bytes = (uint32_t)(min(a.gsegs, a.kst32 - grp * a.gsegs) * kSegBytes);
            mbar_arrive_expect_tx(&fullR[lslot], bytes);
            bulk_g2s(ring + lslot * kF64Rows * row_bytes,
                     a.dig + (int64_t)(src < 0 ? a.zero_cell : src) * cell_bytes +
                         (int64_t)grp * a.gsegs * kSegBytes,
                     bytes, &fullR[lslot]);
            if (++lslot == a.ring) lslot = 0;
            r_issued = ++issued;
            if (++lo == loads) {
                lo = 0;
                lidx += stride;
                src = nsrc;
                nsrc = -1;
                if (f64_work<MODE>(a, li, lidx + stride, count, split, w)) nsrc = f64_source<MODE>(a, w, row);
            }
        };
        for (int k = 0; k < a.ring; ++k) issue();
        int sa = 0, pa = 1, used = 0;  // A stage and phase, the item's first load
        bool ok = true;
        for (int idx = first; ok && idx < count; idx += stride, used += loads) {
            for (int c = 0; ok && c < nch; ++c) {
                for (int grp = 0; ok && grp < groups; ++grp) {
                    const int id = used + (a.resident ? grp : c * groups + grp);
                    const int slot = id % a.ring;
                    ok = mbar_wait_warp(&fullR[slot], (id / a.ring) & 1, abort_v);
                    const unsigned char* mine = ring + slot * kF64Rows * row_bytes;
                    const int ks0 = grp * a.gsegs * 2, ks1 = min(a.ksteps, ks0 + a.gsegs * 2);
#pragma unroll 1
                    for (int ks = ks0; ok && ks < ks1; ++ks) {
                        const unsigned char* at = mine + ((ks - ks0) >> 1) * kSegBytes + (ks & 1) * 16;
                        uint4 b[kDig];
#pragma unroll
                        for (int i = 0; i < kDig; ++i)
                            b[i] = *reinterpret_cast<const uint4*>(at + i * 32);
                        ok = mbar_wait_warp(&emptyA[sa], pa, abort_v);
                        if (!ok) break;
                        tc_fence_after();
#pragma unroll
                        for (int i = 0; i < kDig; ++i) {
                            uint32_t h[8];
                            expand16(b[i], h);
                            tmem_st8(tq + (uint32_t)(sa * kDig * 8 + 8 * i), h);
                        }
                        tmem_wait_st();
                        tc_fence_before();
                        mbar_arrive(&fullA[sa]);
                        if (++sa == kAStages) {
                            sa = 0;
                            pa ^= 1;
                        }
                    }
                    if (!a.resident || c + 1 == nch) {
                        ++freed;
                        issue();
                    }
                }
            }
        }
        if (!ok) *abort_v = 1;
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 (row =
        // lane), warps 0..3 the first half of a chunk's columns, 4..7 the rest
        const int quad = warp & 3, half = warp >> 2, row = quad * 32 + lane;
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16);
        int jacc = 0;
        F64Work w;
        bool stop = false;
        for (int idx = first; !stop && f64_work<MODE>(a, li, idx, count, split, w); idx += stride) {
            const int src = f64_source<MODE>(a, w, row);
            const int er = src >= 0 ? a.rexp[src] : 0;
            const bool fast = abs(er) <= kExpFast - 150;  // operator exponents lie within +-100
            double* orow = a.out + (int64_t)(w.base + row) * a.out_stride;
            for (int c = w.c0; c < w.c1; ++c, ++jacc) {
                const int N = min(kChunk, a.npad - c * kChunk);
                const int ng = N / 8, c0 = half * (N / 2);  // groups of 4 columns
                const int n0 = c * kChunk + c0;
                const int16_t* fe = a.oexp + (int64_t)w.op * a.npad + n0;
                int2 f[6];
#pragma unroll
                for (int q = 0; q < 6; ++q)
                    if (q < ng) f[q] = __ldg(reinterpret_cast<const int2*>(fe) + q);
                int ok = 1;
                if (lane == 0) ok = mbar_wait_or_abort(&accf, jacc & 1, abort_v) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) {
                    *abort_v = 1;
                    stop = true;
                    break;
                }
                tc_fence_after();
                F64Sum I[6][4];
                uint32_t big = 0;  // bits 23 and up set by a sum of 2^22 or more
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    if (q >= ng) break;  // uniform
                    uint32_t s[kAcc][4];
#pragma unroll
                    for (int d = 0; d < kAcc; ++d)
                        tmem_ld4_nw(tq + (uint32_t)(d * kChunk + c0 + 4 * q), s[d]);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 4; ++j) {
                        // s + 1.5 2^23 holds the integer s in its low bits
                        // while |s| < 2^22 (crystals stay below 2^20); the
                        // conversion instruction runs at 16 a clock, the add at 128
                        uint32_t v[kAcc];
#pragma unroll
                        for (int d = 0; d < kAcc; ++d) {
                            v[d] = __float_as_uint(__uint_as_float(s[d][j]) + 12582912.f);
                            big |= v[d] ^ 0x4B400000u;
                        }
                        I[q][j] = f64_join(v);
                    }
                    if (__any_sync(0xffffffffu, big >> 23)) {
                        // (uniform, rare) larger sums by conversion
#pragma unroll 1
                        for (int j = 0; j < 4; ++j) {
                            long long S[2] = {0, 0};
#pragma unroll 1
                            for (int d = 0; d < kAcc; ++d) {
                                uint32_t x[1];
                                tmem_ld1(tq + (uint32_t)(d * kChunk + c0 + 4 * q + j), x);
                                S[d >> 2] = S[d >> 2] * 256 + (long long)__float2int_rn(__uint_as_float(x[0]));
                            }
#pragma unroll
                            for (int jj = 0; jj < 4; ++jj)
                                if (jj == j) I[q][jj] = f64_sum(S[0], S[1]);
                        }
                        big = 0;
                    }
                }
                tc_fence_before();
                mbar_arrive(&acce);  // the issuer may start the next chunk
#pragma unroll
                for (int q = 0; q < 6; ++q) {
                    if (q >= ng) break;
                    if (row >= w.rows) continue;
                    const int fn[4] = {(int)(int16_t)(f[q].x & 0xffff), f[q].x >> 16,
                                       (int)(int16_t)(f[q].y & 0xffff), f[q].y >> 16};
                    double v[4];
                    if (fast) {
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] = fixed_to_double(I[q][j], er + fn[j] - kSumExp);
                    } else {
#pragma unroll
                        for (int j = 0; j < 4; ++j) v[j] = fixed_to_double_slow(I[q][j], er, fn[j] - kSumExp);
                    }
                    // rows are multiples of 4 doubles apart: whole 32-byte units
                    const int n = n0 + 4 * q;
                    if (n >= a.ld) break;
                    double4_32a* o = reinterpret_cast<double4_32a*>(orow + n);
                    double4_32a r = make_double4_32a(v[0], v[1], v[2], v[3]);
                    if (MODE == F64_L2L) {
                        const double4_32a own = *o;
                        // the parent's L_0 reaches the child's L_0 only, as L_0 / 2: it has no digits
                        if (n == 0) r.x += 0.5 * a.up[(int64_t)src * a.ld];
                        r.x += own.x;
                        r.y += own.y;
                        r.z += own.z;
                        r.w += own.w;
                    }
                    *o = r;
                }
            }
        }
    }

    __syncthreads();
    if (*abort_v) {
        // drain (bounded): the products in flight and every copy still owed
        if (warp == 9) mma_drain(&drain_bar);
        if (tid == 8 * 32) {
            for (int s = 0; s < kBStages; ++s)
                if (b_par[s] >= 0) mbar_wait(&fullB[s], (uint32_t)b_par[s]);
            atomicOr(a.err, ERR_TIMEOUT);
        }
        if (warp >= 10)
            for (int k = max(0, r_issued - a.ring); k < r_issued; ++k)
                mbar_wait(&fullR[k % a.ring], (uint32_t)((k / a.ring) & 1));
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                     : "memory");
}

// ---- slicing ------------------------------------------------------------------
// biased exponent field of |v| (1 for zeros and subnormals)
__device__ __forceinline__ int exp_field(double v) {
    const int e = (__double2hiint(v) >> 20) & 0x7ff;
    return e > 0 ? e : 1;
}
// v as X = v 2^(1076 - emax), rounded to nearest (emax >= v's exponent field:
// |X| <= 2^54); integer units only
__device__ __forceinline__ long long fixed54(double v, int emax) {
    const unsigned long long b = (unsigned long long)__double_as_longlong(v);
    const int e = (int)((b >> 52) & 0x7ff);
    unsigned long long m = b & 0xfffffffffffffull;
    if (e > 0) m |= 1ull << 52;
    const int sh = emax - (e > 0 ? e : 1);
    m <<= 1;
    if (sh > 0) m = sh < 56 ? (m + (1ull << (sh - 1))) >> sh : 0ull;
    return (b >> 63) ? -(long long)m : (long long)m;
}

constexpr int kSliceThreads = 256;
constexpr int kSliceRegs = ((kMaxOrder + 1) * (kMaxOrder + 1) + 31) / 32;

// a warp writes the digits of one row, lane l holding coefficients l + 32 r
__device__ __forceinline__ void store_digits(const double (&v)[kSliceRegs], int P, int lane,
                                             uint8_t* dig, int* rexp) {
    int emax = 0;
#pragma unroll
    for (int r = 0; r < kSliceRegs; ++r)
        if (lane + 32 * r < P) emax = max(emax, exp_field(v[r]));
    for (int o = 16; o > 0; o >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, o));
    if (lane == 0) *rexp = emax == 0x7ff ? kRowNan : emax - 1023;
#pragma unroll
    for (int r = 0; r < kSliceRegs; ++r) {
        const int k = lane + 32 * r;
        if (k >= P) break;
        long long X = emax == 0x7ff ? 0ll : fixed54(v[r], emax);
        uint8_t* d = dig + (k >> 5) * kSegBytes + lane;  // [k / 32][digit][k % 32]
#pragma unroll
        for (int s = kDig - 1; s > 0; --s) {
            const long long t = X + 128;
            d[s * 32] = (uint8_t)(t & 255);
            X = t >> 8;
        }
        d[0] = (uint8_t)(X + 128);
    }
}

// digits of the rows of Y (M or L) of one level's cells, k0 = 1: without their
// first coefficient
__global__ void __launch_bounds__(kSliceThreads) k_f64_slice(int level, int k0, int P, int ld, int lda,
                                                             const LevelInfo* linfo,
                                                             const double* __restrict__ Y,
                                                             uint8_t* dig, int* rexp) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int g0 = linfo->gbase[level], g1 = linfo->gbase[level + 1];
    for (int g = g0 + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); g < g1;
         g += (gridDim.x * blockDim.x) >> 5) {
        double v[kSliceRegs];
#pragma unroll
        for (int r = 0; r < kSliceRegs; ++r)
            v[r] = lane + 32 * r >= k0 && lane + 32 * r < P ? Y[(int64_t)g * ld + lane + 32 * r] : 0.0;
        store_digits(v, P, lane, dig + (int64_t)g * kDig * lda, rexp + g);
    }
}

// M of one level's cells = the sum of their children's shifted multipoles
// (rows of Y, octants in order), and its digits
__global__ void __launch_bounds__(kSliceThreads) k_f64_parents(
    int level, int P, int ld, int lda, const LevelInfo* linfo, const uint32_t* __restrict__ code,
    const int32_t* __restrict__ cid, int64_t off_child, const double* __restrict__ Y, double* M,
    uint8_t* dig, int* rexp) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    const int g0 = linfo->gbase[level], g1 = linfo->gbase[level + 1];
    for (int g = g0 + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); g < g1;
         g += (gridDim.x * blockDim.x) >> 5) {
        const int mine = lane < 8 ? cid[off_child + (((int64_t)code[g] << 3) | lane)] : -1;
        double v[kSliceRegs];
#pragma unroll
        for (int r = 0; r < kSliceRegs; ++r) v[r] = 0.0;
        for (int o = 0; o < 8; ++o) {
            const int gc = __shfl_sync(0xffffffffu, mine, o);
            if (gc < 0) continue;
#pragma unroll
            for (int r = 0; r < kSliceRegs; ++r)
                if (lane + 32 * r < P) v[r] += Y[(int64_t)gc * ld + lane + 32 * r];
        }
#pragma unroll
        for (int r = 0; r < kSliceRegs; ++r)
            if (lane + 32 * r < P) M[(int64_t)g * ld + lane + 32 * r] = v[r];
        store_digits(v, P, lane, dig + (int64_t)g * kDig * lda, rexp + g);
    }
}

// Packed operator digits: a warp per (operator, output row n), rows n >= P
// and columns k >= P zero.  T is row-major [n][k] (M2L, L2L) or transposed
// (M2M).
__global__ void __launch_bounds__(256) k_f64_pack(int op0, int nops, int P, int npad, int kst32,
                                                  int transposed, const double* __restrict__ T,
                                                  unsigned char* ops, int64_t op_bytes,
                                                  int16_t* oexp) {
    const int lane = threadIdx.x & 31;
    for (int64_t u = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) >> 5; u < (int64_t)nops * npad;
         u += ((int64_t)gridDim.x * blockDim.x) >> 5) {
        const int o = (int)(u / npad), n = (int)(u % npad);
        const double* To = T + (int64_t)o * P * P;
        double v[kSliceRegs];
        int emax = 0;
#pragma unroll
        for (int r = 0; r < kSliceRegs; ++r) {
            const int k = lane + 32 * r;
            v[r] = 0.0;
            if (n < P && k < P) {
                v[r] = transposed ? To[(int64_t)k * P + n] : To[(int64_t)n * P + k];
                emax = max(emax, exp_field(v[r]));
            }
        }
        for (int d = 16; d > 0; d >>= 1) emax = max(emax, __shfl_xor_sync(0xffffffffu, emax, d));
        if (lane == 0) oexp[(int64_t)(op0 + o) * npad + n] = (int16_t)(emax > 0 ? emax - 1023 : 0);
        const int c = n / kChunk, nc = min(kChunk, npad - c * kChunk), rr = n - c * kChunk;
        unsigned char* img = ops + (int64_t)(op0 + o) * op_bytes +
                             (int64_t)kst32 * kDig * 64 * (c * kChunk);
#pragma unroll
        for (int r = 0; r < kSliceRegs; ++r) {
            const int k = lane + 32 * r;
            if (k >= kst32 * 32) break;
            long long X = emax > 0 ? fixed54(v[r], emax) : 0ll;
            const int kk = k & 31;
            unsigned char* at = img + (int64_t)(k >> 5) * kDig * nc * 64 + (rr >> 3) * 512 +
                                (rr & 7) * 64 + (((kk >> 3) ^ ((rr & 7) >> 1)) << 4) + (kk & 7) * 2;
#pragma unroll
            for (int s = kDig - 1; s >= 0; --s) {
                const long long t = X + 128;
                const int d = s > 0 ? (int)(t & 255) - 128 : (int)X;
                *reinterpret_cast<__half*>(at + s * nc * 64) = __int2half_rn(d);
                X = t >> 8;
            }
        }
    }
}

// bytes of a ring slot of g K segments
int f64_slot(int g) { return kF64Rows * (g * kSegBytes + 16); }
constexpr int kF64SmemMax = 227 * 1024 - 3 * 1024;

int f64_smem(const F64Args& a) {
    return a.bst * kDig * std::min(kChunk, a.npad) * 64 + f64_slot(a.gsegs) * a.ring + 1024;
}

// Shared memory: an item's digits resident in two (or a multiple of) slots
// where they fit beside two B stages (p <= 12), else two slots of three
// segments, streamed; the rest to B stages.  The streamed rows are bound by the
// number of bulk copies (one a row and slot), not by their bytes: M2L at 1e5
// ions, p = 16, with five slots of one segment 21.9 ms, three of two 18.1, two
// of three 17.7; 1,000 ions 450, 368 and 338 us.
void f64_rings(F64Args& a) {
    const int half = (a.kst32 + 1) / 2, groups = (a.kst32 + half - 1) / half;
    a.gsegs = half;
    a.bst = 2;
    a.ring = groups;
    a.resident = f64_smem(a) <= kF64SmemMax ? 1 : 0;
    if (!a.resident) {
        a.gsegs = 3;
        a.ring = 2;
    }
    while (a.bst < kBStages) {
        ++a.bst;
        if (f64_smem(a) > kF64SmemMax) {
            --a.bst;
            break;
        }
    }
    while (a.resident && a.ring + groups < kMaxRing) {
        a.ring += groups;
        if (f64_smem(a) > kF64SmemMax) {
            a.ring -= groups;
            break;
        }
    }
}

F64Args f64_args(const Workspace& ws) {
    F64Args a;
    memset(&a, 0, sizeof a);
    a.P = ws.P;
    a.ld = ws.ld;
    a.lda = m2l_f64_lda(ws.p);
    a.npad = (ws.P + 15) / 16 * 16;
    a.ksteps = (ws.P + 15) / 16;
    a.kst32 = (ws.P + 31) / 32;
    a.nch = (a.npad + kChunk - 1) / kChunk;
    a.op_bytes = (int64_t)a.kst32 * kDig * a.npad * 64;
    f64_rings(a);
    a.zero_cell = ws.cells_max;
    a.dig = ws.f64_dig;
    a.rexp = ws.f64_rexp;
    a.ops = (const unsigned char*)ws.T_f64;
    a.oexp = (const int16_t*)(a.ops + (int64_t)kF64Ops * a.op_bytes);
    a.linfo = ws.linfo;
    a.code = ws.code;
    a.cid = ws.cid;
    a.err = ws.err;
    return a;
}

unsigned f64_grid(const Workspace& ws, int64_t items) {
    int64_t g = ws.m2l_ctas > 0 ? std::min(ws.m2l_ctas, ws.sms) : ws.sms;
    return (unsigned)std::max<int64_t>(1, std::min(g, items));
}

unsigned slice_grid(int64_t rows) {
    const int64_t per = kSliceThreads / 32;
    return (unsigned)std::max<int64_t>(1, std::min<int64_t>((rows + per - 1) / per, 152 * 8));
}

}  // namespace

int m2l_f64_lda(int p) { return ((p + 1) * (p + 1) + 31) / 32 * 32; }

size_t m2l_f64_digit_bytes(int p, int64_t cells) {
    return (size_t)(cells + 1) * kDig * m2l_f64_lda(p);  // and one cell of zeros
}

size_t m2l_f64_operator_bytes(int p) {
    const int64_t P = (p + 1) * (p + 1), npad = (P + 15) / 16 * 16, k32 = (P + 31) / 32;
    return (size_t)kF64Ops * (size_t)(k32 * kDig * npad * 64 + npad * 2);
}

cudaError_t m2l_f64_init() {
    for (const void* f : {(const void*)k_f64_mma<F64_PAIR>, (const void*)k_f64_mma<F64_M2M>,
                          (const void*)k_f64_mma<F64_L2L>}) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                             kF64SmemMax);
        if (e != cudaSuccess) return e;
    }
    return cudaSuccess;
}

cudaError_t m2l_f64_pack(const Workspace& ws) {
    const F64Args a = f64_args(ws);
    struct Set {
        int op0, n, tr;
        const void* T;
    };
    for (const Set& s : {Set{0, 343, 0, ws.T_m2l}, Set{kF64M2M, 8, 1, ws.T_m2m},
                         Set{kF64L2L, 8, 0, ws.T_l2l}}) {
        k_f64_pack<<<152 * 8, 256>>>(s.op0, s.n, a.P, a.npad, a.kst32, s.tr, (const double*)s.T,
                                     (unsigned char*)ws.T_f64, a.op_bytes, (int16_t*)a.oexp);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaStreamSynchronize(0);
}

static cudaError_t slice(int64_t n, int l, int k0, const double* Y, Workspace& ws, cudaStream_t s) {
    return launch_pdl(k_f64_slice, dim3(slice_grid(level_cap(n, l))), dim3(kSliceThreads), 0, s, l, k0,
                      ws.P, ws.ld, m2l_f64_lda(ws.p), (const LevelInfo*)ws.linfo, Y, ws.f64_dig,
                      ws.f64_rexp);
}
cudaError_t launch_f64_slice(int64_t n, int l, const double* M, Workspace& ws, cudaStream_t s) {
    return slice(n, l, 0, M, ws, s);
}

cudaError_t launch_f64_m2m(int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    const DenseLayout dl = dense_layout(D);
    F64Args a = f64_args(ws);
    a.level = l + 1;  // the children, each row its own shifted multipole in L
    a.out = (double*)ws.L;
    a.out_stride = ws.ld;
    const int64_t items = (level_cap(n, l + 1) / kF64Rows + 8) * a.nch;
    cudaError_t e = launch_pdl(k_f64_mma<F64_M2M>, dim3(f64_grid(ws, items)), dim3(kF64Threads),
                               f64_smem(a), s, a);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_f64_parents, dim3(slice_grid(level_cap(n, l))), dim3(kSliceThreads), 0, s, l,
                      ws.P, ws.ld, a.lda, (const LevelInfo*)ws.linfo, (const uint32_t*)ws.code,
                      (const int32_t*)ws.cid, dl.off[l + 1], (const double*)ws.L, (double*)ws.M,
                      ws.f64_dig, ws.f64_rexp);
}

cudaError_t launch_f64_l2l(int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    cudaError_t e = slice(n, l - 1, 1, (const double*)ws.L, ws, s);
    if (e != cudaSuccess) return e;
    F64Args a = f64_args(ws);
    a.level = l;
    a.off_parent = dense_layout(D).off[l - 1];
    a.up = (const double*)ws.L;
    a.out = (double*)ws.L;
    a.out_stride = ws.ld;
    const int64_t items = (level_cap(n, l) / kF64Rows + 8) * a.nch;
    return launch_pdl(k_f64_mma<F64_L2L>, dim3(f64_grid(ws, items)), dim3(kF64Threads),
                      f64_smem(a), s, a);
}

cudaError_t launch_f64_m2l(Workspace& ws, cudaStream_t s) {
    const PairList L = pair_list(ws);
    F64Args a = f64_args(ws);
    a.hdr = L.hdr;
    a.items = L.items;
    a.pairs = L.pairs;
    a.out = (double*)ws.pp_part;
    a.out_stride = ws.pp_stride;
    k_f64_mma<F64_PAIR><<<f64_grid(ws, ws.pp_item_cap * a.nch), kF64Threads, f64_smem(a), s>>>(a);
    return cudaGetLastError();
}

}  // namespace pt
