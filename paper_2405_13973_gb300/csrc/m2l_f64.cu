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
//     have one weight, so they share an accumulator s_{i+j}, i + j = 0 .. 6:
//     28 products; i + j >= 7 lies below 2^-53 of the product of the two
//     maxima.  |s_d| <= ((d - 1) + 1) 2^14 P for d >= 1 stays below 2^24 for
//     d <= 5 at p = 12 and d <= 3 at p = 16; beyond that bound (which needs
//     every digit at its limit: 2^20 is what crystals reach) the last bit of
//     s_d would be rounded, 2^-45 of the product of the maxima or less;
//   * S = sum_d s_d 2^(8 (6 - d)) is formed in 64-bit integers (its lowest 8
//     bits rounded away) and written as a double: the FP64 units, two lanes
//     per clock and SM, take no part.
// Against a long double sum the result is as good as FP64 multiply-adds
// (2e-16 .. 2e-15 of the row's norm, p = 4 .. 16).
//
// One CTA per SM walks the work items (one operator, up to 128 rows):
//   D[128 rows x N] = sum over K steps of 16, i, j:  A_i[128 x 16] B_j[16 x N],
// in column chunks of up to 48 outputs so that the seven accumulators (336
// TMEM columns) leave room for three K steps of A in tensor memory (7 digits
// x 8 columns each).  A comes from tensor memory because with 48 columns a
// product takes 24 cycles and reading a 4 KB A tile from shared memory 32:
//   * warps 10..13 (one TMEM lane quarter each) load the rows' digits (one
//     byte per digit and coefficient: half the bytes of f16, and the digits
//     of an item, 172 KB at p = 12, are read once per column chunk, mostly
//     from L1), expand them to f16 (a byte permute into 1024 + d + 128, one
//     packed subtraction) and store them to tensor memory;
//   * warp 8 brings the operator digits, packed in f16 in the swizzled
//     K-major shared-memory image, by bulk copies of 32-wide K chunks;
//   * warp 9 issues the 28 products of a K step;
//   * warps 0..7 read the accumulators, release them once the integers are
//     formed, and write the doubles while the next chunk's products run.
// Every mbarrier wait is bounded as in m2l_tc.cu.
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
constexpr int kAStages = 3;             // K steps of A in tensor memory
constexpr int kACol0 = kDig * kChunk;   // their first TMEM column
constexpr int kBStages = 4;             // 32-wide K chunks of B in shared memory
constexpr int kF64Threads = 448;
constexpr int kF64Ops = 359;            // 343 M2L offsets, 8 M2M, 8 L2L octants
constexpr int kF64M2M = 343, kF64L2L = 351;
constexpr int kRowNan = 0x7fffffff;     // exponent of a row with a NaN or infinity

enum F64Mode { F64_PAIR = 0, F64_M2M = 1, F64_L2L = 2 };

struct F64Args {
    int P, ld, lda;            // coefficients, row stride of M, L and partial rows, digit row stride
    int npad, ksteps, kst32, nch, level, sms;
    int64_t out_stride, op_bytes;
    const uint8_t* dig;        // [cell][kDig][lda]
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
    double* out;
    int* err;
};

// instruction descriptor: D f32, A and B f16, K-major
__device__ __forceinline__ uint32_t idesc_f16(int N) {
    return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(kF64Rows >> 4) << 24);
}
__device__ __forceinline__ void mma_f16_ts(uint32_t dtmem, uint32_t atmem, uint64_t bd,
                                           uint32_t idesc, uint32_t accum) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n}" ::"r"(dtmem),
        "r"(atmem), "l"(bd), "r"(idesc), "r"(accum)
        : "memory");
}
__device__ __forceinline__ void tmem_ld8_nw(uint32_t taddr, uint32_t (&r)[8]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
          "=r"(r[7])
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

// I 2^e as a double, rounded to nearest, without the FP64 units
__device__ __forceinline__ double fixed_to_double(long long I, int e) {
    if (I == 0) return 0.0;
    const unsigned long long a = I < 0 ? 0ull - (unsigned long long)I : (unsigned long long)I;
    const int lz = __clzll((long long)a);
    const unsigned long long m = a << lz;
    const int be = e + 63 - lz + 1022;  // exponent field before the hidden bit is added
    if (be < 1 || be > 2044) return ldexp((double)I, e);
    const unsigned long long r = ((unsigned long long)be << 52) + (m >> 11) + ((m >> 10) & 1ull);
    return __longlong_as_double((long long)(r | ((unsigned long long)I & 0x8000000000000000ull)));
}

// work item idx: operator, rows, and for M2M / L2L the first target cell
struct F64Work {
    int op, rows, base;
};
template <int MODE>
__device__ __forceinline__ bool f64_work(const F64Args& a, const LevelInfo& li, int idx, int count,
                                         F64Work& w) {
    w.rows = 0;
    w.op = 0;
    w.base = 0;
    if (idx >= count) return false;
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
        emptyB[kBStages], accf, acce, drain_bar;
    __shared__ uint32_t tmem_base_sh;
    __shared__ int abort_sh;
    __shared__ LevelInfo li;
    volatile int* abort_v = &abort_sh;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
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
        mbar_init(&accf, 1);
        mbar_init(&acce, 256);
        mbar_init(&drain_bar, 1);
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    __syncthreads();
    const int count = f64_count<MODE>(a, li);
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
    int b_par[kBStages];  // operator producer: parity of the last copy per stage
#pragma unroll
    for (int s = 0; s < kBStages; ++s) b_par[s] = -1;

    if (warp == 8) {
        // ---- operator producer
        if (lane == 0) {
            int g = 0;
            F64Work w;
            for (int idx = first; f64_work<MODE>(a, li, idx, count, w) && !*abort_v; idx += stride) {
                const unsigned char* src = a.ops + (int64_t)w.op * a.op_bytes;
                for (int c = 0; c < a.nch; ++c) {
                    const uint32_t bytes = (uint32_t)(kDig * min(kChunk, a.npad - c * kChunk) * 64);
                    for (int k = 0; k < a.kst32; ++k, ++g) {
                        const int st = g % kBStages, use = g / kBStages;
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
        // ---- MMA issuer
        if (lane == 0) {
            int ga = 0, gb = 0, jacc = 0;
            F64Work w;
            for (int idx = first; f64_work<MODE>(a, li, idx, count, w) && !*abort_v; idx += stride) {
                for (int c = 0; c < a.nch && !*abort_v; ++c, ++jacc) {
                    const int N = min(kChunk, a.npad - c * kChunk);
                    const uint32_t id = idesc_f16(N);
                    const uint64_t bstep = (uint64_t)((N * 64) >> 4);  // one digit of B
                    // the epilogue has read the previous chunk's accumulators
                    if (jacc > 0 && !mbar_wait_or_abort(&acce, (jacc - 1) & 1, abort_v)) {
                        *abort_v = 1;
                        break;
                    }
                    for (int ks = 0; ks < a.ksteps; ++ks, ++ga) {
                        const int sb = gb % kBStages, ub = gb / kBStages;
                        const int sa = ga % kAStages, ua = ga / kAStages;
                        if (!(ks & 1) && !mbar_wait_or_abort(&fullB[sb], ub & 1, abort_v)) {
                            *abort_v = 1;
                            break;
                        }
                        if (!mbar_wait_or_abort(&fullA[sa], ua & 1, abort_v)) {
                            *abort_v = 1;
                            break;
                        }
                        tc_fence_after();
                        const uint64_t bd = sdesc64(smem_addr(base + sb * b_stage) + 32u * (ks & 1));
                        const uint32_t at = tmem + (uint32_t)(kACol0 + sa * kDig * 8);
                        const uint32_t more = ks > 0 ? 1u : 0u;
#pragma unroll
                        for (int i = 0; i < kDig; ++i)
#pragma unroll
                            for (int j = 0; j + i < kDig; ++j)
                                mma_f16_ts(tmem + (uint32_t)((i + j) * kChunk), at + (uint32_t)(8 * i),
                                           bd + bstep * (uint64_t)j, id, i > 0 ? 1u : more);
                        mma_commit(&emptyA[sa]);
                        if ((ks & 1) || ks + 1 == a.ksteps) {
                            mma_commit(&emptyB[sb]);
                            ++gb;
                        }
                    }
                    if (*abort_v) break;
                    mma_commit(&accf);
                }
            }
        }
    } else if (warp >= 10) {
        // ---- A producers: thread = row; a K step's seven digit groups (16
        // bytes each) are loaded two steps ahead of their expansion
        const int quad = warp & 3, row = quad * 32 + lane;
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16) + (uint32_t)kACol0;
        const int64_t cell_bytes = (int64_t)kDig * a.lda;
        int idx = first, c = 0, k = 0;  // the next step to load
        F64Work w;
        bool more = f64_work<MODE>(a, li, idx, count, w);
        int src = more ? f64_source<MODE>(a, w, row) : -1, nsrc = -1;
        if (f64_work<MODE>(a, li, idx + stride, count, w)) nsrc = f64_source<MODE>(a, w, row);
        auto load = [&](uint4 (&b)[kDig]) {
            if (!more) return;
            const uint8_t* p = a.dig + (int64_t)(src < 0 ? 0 : src) * cell_bytes + 16 * k;
#pragma unroll
            for (int i = 0; i < kDig; ++i)
                b[i] = src >= 0 ? __ldg(reinterpret_cast<const uint4*>(p + i * a.lda))
                                : make_uint4(0x80808080u, 0x80808080u, 0x80808080u, 0x80808080u);
            if (++k == a.ksteps) {
                k = 0;
                if (++c == a.nch) {
                    c = 0;
                    idx += stride;
                    more = idx < count;
                    src = nsrc;
                    nsrc = -1;
                    if (f64_work<MODE>(a, li, idx + stride, count, w))
                        nsrc = f64_source<MODE>(a, w, row);
                }
            }
        };
        int g = 0;
        auto store = [&](const uint4 (&b)[kDig]) -> bool {
            const int st = g % kAStages, use = g / kAStages;
            ++g;
            int ok = 1;
            if (lane == 0) ok = mbar_wait_or_abort(&emptyA[st], (use & 1) ^ 1, abort_v) ? 1 : 0;
            ok = __shfl_sync(0xffffffffu, ok, 0);
            if (!ok) {
                *abort_v = 1;
                return false;
            }
            tc_fence_after();
#pragma unroll
            for (int i = 0; i < kDig; ++i) {
                uint32_t h[8];
                expand16(b[i], h);
                tmem_st8(tq + (uint32_t)(st * kDig * 8 + 8 * i), h);
            }
            tmem_wait_st();
            tc_fence_before();
            mbar_arrive(&fullA[st]);
            return true;
        };
        uint4 b0[kDig], b1[kDig];
        bool h0 = more;
        load(b0);
        bool h1 = more;
        load(b1);
        while (h0) {
            if (!store(b0)) break;
            h0 = more;
            load(b0);
            if (!h1 || !store(b1)) break;
            h1 = more;
            load(b1);
        }
    } else {
        // ---- epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 (row =
        // lane), warps 0..3 the first half of a chunk's columns, 4..7 the rest
        const int quad = warp & 3, half = warp >> 2, row = quad * 32 + lane;
        const uint32_t tq = tmem + ((uint32_t)(quad * 32) << 16);
        int jacc = 0;
        F64Work w;
        bool stop = false;
        for (int idx = first; !stop && f64_work<MODE>(a, li, idx, count, w); idx += stride) {
            const int src = f64_source<MODE>(a, w, row);
            const int er = src >= 0 ? a.rexp[src] : 0;
            double* orow = a.out + (int64_t)(w.base + row) * a.out_stride;
            for (int c = 0; c < a.nch; ++c, ++jacc) {
                const int N = min(kChunk, a.npad - c * kChunk);
                const int ng = N / 16, c0 = half * (N / 2);  // groups of 8 columns
                const int n0 = c * kChunk + c0;
                const int16_t* fe = a.oexp + (int64_t)w.op * a.npad + n0;
                int4 f[3];
#pragma unroll
                for (int q = 0; q < 3; ++q)
                    if (q < ng) f[q] = __ldg(reinterpret_cast<const int4*>(fe) + q);
                int ok = 1;
                if (lane == 0) ok = mbar_wait_or_abort(&accf, jacc & 1, abort_v) ? 1 : 0;
                ok = __shfl_sync(0xffffffffu, ok, 0);
                if (!ok) {
                    *abort_v = 1;
                    stop = true;
                    break;
                }
                tc_fence_after();
                long long I[3][8];
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if (q >= ng) break;  // uniform
                    uint32_t s[kDig][8];
#pragma unroll
                    for (int d = 0; d < kDig; ++d)
                        tmem_ld8_nw(tq + (uint32_t)(d * kChunk + c0 + 8 * q), s[d]);
                    tmem_wait_ld();
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        int v[kDig];
#pragma unroll
                        for (int d = 0; d < kDig; ++d) v[d] = __float2int_rn(__uint_as_float(s[d][j]));
                        const long long hi = (long long)v[0] * (1 << 24) +
                                             ((long long)v[1] * (1 << 16) +
                                              ((long long)v[2] * (1 << 8) + (long long)v[3]));
                        const long long lo = (long long)v[4] * (1 << 16) +
                                             ((long long)v[5] * (1 << 8) + (long long)v[6]);
                        I[q][j] = (hi << 16) + ((lo + 128) >> 8);
                    }
                }
                tc_fence_before();
                mbar_arrive(&acce);  // the issuer may start the next chunk
#pragma unroll
                for (int q = 0; q < 3; ++q) {
                    if (q >= ng) break;
                    if (row >= w.rows) continue;
                    const int fw[4] = {f[q].x, f[q].y, f[q].z, f[q].w};
                    double v[8];
#pragma unroll
                    for (int j = 0; j < 8; ++j) {
                        const int fn = j & 1 ? fw[j >> 1] >> 16 : (int)(int16_t)(fw[j >> 1] & 0xffff);
                        v[j] = er == kRowNan ? __longlong_as_double(0x7ff8000000000000ll)
                                             : fixed_to_double(I[q][j], er + fn - 50);
                    }
                    // rows are multiples of 4 doubles apart: whole 32-byte units
#pragma unroll
                    for (int u = 0; u < 2; ++u) {
                        const int n = n0 + 8 * q + 4 * u;
                        if (n >= a.ld) break;
                        double4_32a* o = reinterpret_cast<double4_32a*>(orow + n);
                        double4_32a r = make_double4_32a(v[4 * u], v[4 * u + 1], v[4 * u + 2], v[4 * u + 3]);
                        if (MODE == F64_L2L) {
                            const double4_32a own = *o;
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
    }

    __syncthreads();
    if (*abort_v) {
        // drain (bounded): the products in flight and every copy still owed
        if (tid == 9 * 32) {
            mma_commit(&drain_bar);
            mbar_wait(&drain_bar, 0);
        }
        if (tid == 8 * 32) {
            for (int s = 0; s < kBStages; ++s)
                if (b_par[s] >= 0) mbar_wait(&fullB[s], (uint32_t)b_par[s]);
            atomicOr(a.err, ERR_TIMEOUT);
        }
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
__device__ __forceinline__ void store_digits(const double (&v)[kSliceRegs], int P, int lane, int lda,
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
#pragma unroll
        for (int s = kDig - 1; s > 0; --s) {
            const long long t = X + 128;
            dig[s * lda + k] = (uint8_t)(t & 255);
            X = t >> 8;
        }
        dig[k] = (uint8_t)(X + 128);
    }
}

// digits of the rows of Y (M or L) of one level's cells
__global__ void __launch_bounds__(kSliceThreads) k_f64_slice(int level, int P, int ld, int lda,
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
            v[r] = lane + 32 * r < P ? Y[(int64_t)g * ld + lane + 32 * r] : 0.0;
        store_digits(v, P, lane, lda, dig + (int64_t)g * kDig * lda, rexp + g);
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
        store_digits(v, P, lane, lda, dig + (int64_t)g * kDig * lda, rexp + g);
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

int f64_smem(int npad) { return kBStages * kDig * std::min(kChunk, npad) * 64 + 1024; }

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

size_t m2l_f64_digit_bytes(int p, int64_t cells) { return (size_t)cells * kDig * m2l_f64_lda(p); }

size_t m2l_f64_operator_bytes(int p) {
    const int64_t P = (p + 1) * (p + 1), npad = (P + 15) / 16 * 16, k32 = (P + 31) / 32;
    return (size_t)kF64Ops * (size_t)(k32 * kDig * npad * 64 + npad * 2);
}

cudaError_t m2l_f64_init() {
    const int smem = f64_smem(kChunk);
    // the rest of the SM's memory as L1: the digit rows are read once per chunk
    const int carve = 45;
    for (const void* f : {(const void*)k_f64_mma<F64_PAIR>, (const void*)k_f64_mma<F64_M2M>,
                          (const void*)k_f64_mma<F64_L2L>}) {
        cudaError_t e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, carve);
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

cudaError_t launch_f64_slice(int64_t n, int l, const double* Y, Workspace& ws, cudaStream_t s) {
    return launch_pdl(k_f64_slice, dim3(slice_grid(level_cap(n, l))), dim3(kSliceThreads), 0, s, l,
                      ws.P, ws.ld, m2l_f64_lda(ws.p), (const LevelInfo*)ws.linfo, Y, ws.f64_dig,
                      ws.f64_rexp);
}

cudaError_t launch_f64_m2m(int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    const DenseLayout dl = dense_layout(D);
    F64Args a = f64_args(ws);
    a.level = l + 1;  // the children, each row its own shifted multipole in L
    a.out = (double*)ws.L;
    a.out_stride = ws.ld;
    const int64_t items = level_cap(n, l + 1) / kF64Rows + 8;
    cudaError_t e = launch_pdl(k_f64_mma<F64_M2M>, dim3(f64_grid(ws, items)), dim3(kF64Threads),
                               f64_smem(a.npad), s, a);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_f64_parents, dim3(slice_grid(level_cap(n, l))), dim3(kSliceThreads), 0, s, l,
                      ws.P, ws.ld, a.lda, (const LevelInfo*)ws.linfo, (const uint32_t*)ws.code,
                      (const int32_t*)ws.cid, dl.off[l + 1], (const double*)ws.L, (double*)ws.M,
                      ws.f64_dig, ws.f64_rexp);
}

cudaError_t launch_f64_l2l(int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    cudaError_t e = launch_f64_slice(n, l - 1, (const double*)ws.L, ws, s);
    if (e != cudaSuccess) return e;
    F64Args a = f64_args(ws);
    a.level = l;
    a.off_parent = dense_layout(D).off[l - 1];
    a.out = (double*)ws.L;
    a.out_stride = ws.ld;
    const int64_t items = level_cap(n, l) / kF64Rows + 8;
    return launch_pdl(k_f64_mma<F64_L2L>, dim3(f64_grid(ws, items)), dim3(kF64Threads),
                      f64_smem(a.npad), s, a);
}

cudaError_t launch_f64_m2l(Workspace& ws, cudaStream_t s) {
    const PairList L = pair_list(ws);
    F64Args a = f64_args(ws);
    a.hdr = L.hdr;
    a.items = L.items;
    a.pairs = L.pairs;
    a.out = (double*)ws.pp_part;
    a.out_stride = ws.pp_stride;
    k_f64_mma<F64_PAIR><<<f64_grid(ws, ws.pp_item_cap), kF64Threads, f64_smem(a.npad), s>>>(a);
    return cudaGetLastError();
}

}  // namespace pt
