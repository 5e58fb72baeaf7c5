// m2l_f32.cu -- the dense FP32 translations (M2M, M2L of Eq. FMM_local, L2L)
// of PT_FP32 plans on the CUDA cores.
//
// Every output is one chain of fused multiply-adds in the order of the terms
// and of the coefficients, out[r][n] = fma(a[r][k], T[n][k], .) for k = 0, 1,
// ..., whatever the tiling; a missing source adds zeros.  Four uses:
//   PAIR  the pair work list: one term (the item's offset), rows = its pairs,
//         each product row to its partial row;
//   TILE  up to 128 targets of one octant of a level: its 189 offsets, then
//         the octant's L2L of the parents (levels >= 3);
//   M2M   parents of a level: the eight octants' children in turn;
//   L2L   children of one octant: their own M2L sum plus the parents' shift.
// Bound by the FP32 pipe.  A block computes 16 R rows x NC columns (all of
// them up to p = 12, two halves above), thread (row group, column group) R x 8
// outputs as packed pairs of columns (fma.rn.f32x2: both halves rounded as by
// fma.rn.f32, at half the issue slots), operands from a three-stage cp.async
// ring of 32-wide K chunks: A rows as they lie in memory, read four
// coefficients at a time and broadcast; B = the transposed operator, packed
// per plan kind as [operator][K][columns], 4 + 4 columns per thread so that
// neighbouring threads read neighbouring 16-byte units.  With 64 x 64 tiles
// of 4 x 4 outputs staged element by element through two barriers per 16
// coefficients the product ran at 16 TFLOP/s (12.0 ms for the 3.35 M pairs of
// the 1e5-ion sphere, p = 12), now at 37 (5.1 ms).  Tiles beyond 262,144 ions: a
// field at 1e6 ions, p = 12, 166 -> 66 ms.
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

constexpr int kRowGroups = 16;
constexpr int kF32Stages = 3;
constexpr int kAStride = 36;      // floats per A row in shared memory (32 + 4: no bank conflicts)
constexpr int kMaxGroups = 22;    // column groups of 8 per block
constexpr int kF32MaxThreads = kRowGroups * kMaxGroups;
constexpr int kF32M2M = 343, kF32L2L = 351, kF32Ops = 359;

enum F32Mode { F32_PAIR = 0, F32_TILE = 1, F32_M2M = 2, F32_L2L = 3 };

// columns: blocks per row tile and columns per block
struct F32Cols {
    int split, nc;
};
__host__ __device__ inline F32Cols f32_cols(int P) {
    const int g = P <= 32 ? 4 : (P + 7) / 8;  // 64 threads at least
    F32Cols c;
    c.split = g > kMaxGroups ? 2 : 1;
    c.nc = 8 * ((g + c.split - 1) / c.split);
    return c;
}

struct F32Args {
    int P, ld, kch, nc, split, level;
    int64_t op_vals;           // kch * 32 * split * nc
    const float* ops;          // [kF32Ops][kch * 32][split][nc]
    const M2lPairHdr* hdr;
    const M2lPairItem* items;
    const M2lPair* pairs;
    const LevelInfo* linfo;
    const uint32_t* code;
    const int32_t* cid;
    int64_t off_level, off_other;  // dense maps: the targets' level; parents (TILE, L2L) or children (M2M)
    const float* M;
    float* L;
    float* out;                // PAIR: partial rows; M2M: M
};

__constant__ int16_t c_f32_off[8][189];

struct F32Unit {
    int row0, rows, oct, op, col;  // first row, rows, octant, PAIR operator, column block
};

// unit u of the launch: (row tile, column block)
template <int MODE, int ROWS>
__device__ __forceinline__ bool f32_unit(const F32Args& a, const LevelInfo& li, int u, F32Unit& w) {
    int t = u / a.split;
    w.col = u - t * a.split;
    if (MODE == F32_PAIR) {
        constexpr int parts = kPairRows / ROWS;
        if (t >= a.hdr->n_items * parts) return false;
        const M2lPairItem it = a.items[t / parts];
        const int r0 = (t % parts) * ROWS;
        w.op = it.op;
        w.row0 = it.begin + r0;
        w.rows = min(ROWS, it.rows - r0);  // may be <= 0: nothing to do
        w.oct = 0;
        return true;
    }
    if constexpr (MODE == F32_M2M) {
        const int g0 = li.gbase[a.level], g1 = li.gbase[a.level + 1];
        w.row0 = g0 + t * ROWS;
        w.rows = min(ROWS, g1 - w.row0);
        w.oct = w.op = 0;
        return w.rows > 0;
    }
    // tiles of one octant's cells
    for (int o = 0; MODE != F32_M2M && o < 8; ++o) {
        const int s0 = li.oct_start[a.level][o], s1 = li.oct_start[a.level][o + 1];
        const int nt = (s1 - s0 + ROWS - 1) / ROWS;
        if (t < nt) {
            w.row0 = s0 + t * ROWS;
            w.rows = min(ROWS, s1 - w.row0);
            w.oct = o;
            w.op = 0;
            return true;
        }
        t -= nt;
    }
    return false;
}
template <int MODE>
__device__ __forceinline__ int f32_terms(const F32Args& a) {
    return MODE == F32_TILE ? 189 + (a.level >= 3 ? 1 : 0) : MODE == F32_M2M ? 8 : 1;
}
template <int MODE>
__device__ __forceinline__ int f32_op(const F32Unit& w, int term) {
    if (MODE == F32_PAIR) return w.op;
    if (MODE == F32_M2M) return kF32M2M + term;
    if (MODE == F32_L2L) return kF32L2L + w.oct;
    return term < 189 ? (int)c_f32_off[w.oct][term] : kF32L2L + w.oct;
}
// the coefficient row that row r of the unit takes in a term, or null
template <int MODE>
__device__ __forceinline__ const float* f32_source(const F32Args& a, const F32Unit& w, int term, int r) {
    if (r >= w.rows) return nullptr;
    if (MODE == F32_PAIR) return a.M + (int64_t)a.pairs[w.row0 + r].src * a.ld;
    const uint32_t c = a.code[w.row0 + r];
    if (MODE == F32_M2M) {
        const int g = a.cid[a.off_other + (((int64_t)c << 3) | term)];
        return g >= 0 ? a.M + (int64_t)g * a.ld : nullptr;
    }
    if (MODE == F32_L2L || term >= 189) {
        const int g = a.cid[a.off_other + (c >> 3)];
        return g >= 0 ? a.L + (int64_t)g * a.ld : nullptr;
    }
    const int op = c_f32_off[w.oct][term], lim = 1 << a.level;
    int x, y, z;
    demorton3(c, x, y, z);
    x -= op / 49 - 3;
    y -= (op / 7) % 7 - 3;
    z -= op % 7 - 3;
    if (x < 0 || y < 0 || z < 0 || x >= lim || y >= lim || z >= lim) return nullptr;
    const int g = a.cid[a.off_level + morton3(x, y, z)];
    return g >= 0 ? a.M + (int64_t)g * a.ld : nullptr;
}

__device__ __forceinline__ unsigned long long pack2(float lo, float hi) {
    unsigned long long r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(unsigned long long v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(unsigned long long& c, unsigned long long x, unsigned long long y) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(c) : "l"(x), "l"(y));
}

// R rows per thread: 8 (tiles of 128 rows), or 2 (32 rows) where a level has
// too few cells to fill the GPU with the larger tiles
template <int MODE, int R>
__global__ void __launch_bounds__(kF32MaxThreads) k_f32_gemm(const __grid_constant__ F32Args a) {
    constexpr int ROWS = kRowGroups * R;
    extern __shared__ __align__(16) float f32_smem[];
    __shared__ const float* s_src[2][ROWS];
    __shared__ LevelInfo li;
    pdl_wait();
    const int tid = threadIdx.x, nthr = blockDim.x;
    const int cgs = a.nc / 8, cg = tid % cgs, rg = tid / cgs;
    const int a_vals = ROWS * kAStride, stage_vals = a_vals + 32 * a.nc;
    if (MODE != F32_PAIR) {
        const int* src = reinterpret_cast<const int*>(a.linfo);
        int* dst = reinterpret_cast<int*>(&li);
        for (int i = tid; i < (int)(sizeof(LevelInfo) / sizeof(int)); i += nthr) dst[i] = src[i];
        __syncthreads();
    }
    const int terms = f32_terms<MODE>(a);
    // the loading side runs kF32Stages - 1 chunks ahead: unit, term, chunk
    int lu = blockIdx.x, lterm = 0, lk = 0, lbuf = 0, lst = 0;
    F32Unit lw;
    bool lmore = f32_unit<MODE, ROWS>(a, li, lu, lw);
    // sources of the term after the one being loaded, by thread = row, in registers
    F32Unit nw = lw;
    int nu = lu, nterm = 0;
    bool nmore = lmore;
    auto advance = [&](int& u, int& term, F32Unit& w, bool& more) {
        if (++term < terms) return;
        term = 0;
        u += gridDim.x;
        more = f32_unit<MODE, ROWS>(a, li, u, w);
    };
    auto fetch = [&](int r) -> const float* {
        return nmore && r < ROWS ? f32_source<MODE>(a, nw, nterm, r) : nullptr;
    };
    constexpr int NSRC = 2;  // rows per thread at most (at least 64 threads)
    const float* nsrc[NSRC];
#pragma unroll
    for (int j = 0; j < NSRC; ++j) {
        const float* p = fetch(tid + j * nthr);
        if (tid + j * nthr < ROWS) s_src[0][tid + j * nthr] = p;
    }
    if (nmore) advance(nu, nterm, nw, nmore);
#pragma unroll
    for (int j = 0; j < NSRC; ++j) nsrc[j] = fetch(tid + j * nthr);
    __syncthreads();
    auto load = [&]() {
        if (lmore) {
            float* sA = f32_smem + lst * stage_vals;
            float* sB = sA + a_vals;
            // a thread's 16-byte unit q is the same in all its rows (nthr is a multiple
            // of 16).  Zeros beyond column P: the rows' padding takes no part,
            // whatever it holds (a row with a NaN leaves NaN there, below)
            const int q = tid & 7, col = lk * 32 + 4 * q;
            const uint32_t bytes = 4u * (uint32_t)max(0, min(4, a.P - col));
            for (int r = tid >> 3; r < ROWS; r += nthr >> 3) {
                const float* src = s_src[lbuf][r];
                cp_async16(sA + r * kAStride + 4 * q, src ? src + col : a.M, src ? bytes : 0u);
            }
            const int rowq = a.nc / 4;  // 16-byte units per K row
            const float* B = a.ops + (int64_t)f32_op<MODE>(lw, lterm) * a.op_vals +
                             ((int64_t)lk * 32 * a.split + lw.col) * a.nc;
            for (int u = tid; u < 32 * rowq; u += nthr) {
                const int k = u / rowq, q = u - k * rowq;
                cp_async16(sB + k * a.nc + 4 * q, B + (int64_t)k * a.split * a.nc + 4 * q, 16u);
            }
            if (++lst == kF32Stages) lst = 0;
            if (++lk == a.kch) {
                lk = 0;
                lbuf ^= 1;
                // read after the barrier before the next load
#pragma unroll
                for (int j = 0; j < NSRC; ++j)
                    if (tid + j * nthr < ROWS) s_src[lbuf][tid + j * nthr] = nsrc[j];
                advance(lu, lterm, lw, lmore);
                if (nmore) advance(nu, nterm, nw, nmore);
#pragma unroll
                for (int j = 0; j < NSRC; ++j) nsrc[j] = fetch(tid + j * nthr);
            }
        }
        cp_async_commit();
    };
    for (int s = 0; s < kF32Stages - 1; ++s) {
        load();
        __syncthreads();
    }
    int st = 0;
    F32Unit w;
    for (int u = blockIdx.x; f32_unit<MODE, ROWS>(a, li, u, w); u += gridDim.x) {
        unsigned long long acc[R][4];
        const int n0 = w.col * a.nc + 4 * cg, n1 = n0 + a.nc / 2;
#pragma unroll
        for (int r = 0; r < R; ++r) {
#pragma unroll
            for (int j = 0; j < 4; ++j) acc[r][j] = 0ull;
            const int row = r * kRowGroups + rg;
            if (MODE == F32_L2L && row < w.rows) {
                const float* own = a.L + (int64_t)(w.row0 + row) * a.ld;
                if (n0 < a.ld) {
                    const float4 v = *reinterpret_cast<const float4*>(own + n0);
                    acc[r][0] = pack2(v.x, v.y);
                    acc[r][1] = pack2(v.z, v.w);
                }
                if (n1 < a.ld) {
                    const float4 v = *reinterpret_cast<const float4*>(own + n1);
                    acc[r][2] = pack2(v.x, v.y);
                    acc[r][3] = pack2(v.z, v.w);
                }
            }
        }
        for (int c = 0; c < terms * a.kch; ++c) {
            cp_async_wait(kF32Stages - 2);
            __syncthreads();  // the chunk is in; the one before is read by all
            load();
            const float* sA = f32_smem + st * stage_vals + rg * kAStride;
            const float* sB = f32_smem + st * stage_vals + a_vals + 4 * cg;
            if (++st == kF32Stages) st = 0;
#pragma unroll 2
            for (int k4 = 0; k4 < 8; ++k4) {
                float4 av[R];
#pragma unroll
                for (int r = 0; r < R; ++r)
                    av[r] = *reinterpret_cast<const float4*>(sA + r * kRowGroups * kAStride + 4 * k4);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk) {
                    const float* bp = sB + (4 * k4 + kk) * a.nc;
                    const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(bp);
                    const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(bp + a.nc / 2);
#pragma unroll
                    for (int r = 0; r < R; ++r) {
                        const float x = kk == 0 ? av[r].x : kk == 1 ? av[r].y : kk == 2 ? av[r].z : av[r].w;
                        const unsigned long long xx = pack2(x, x);
                        fma2(acc[r][0], xx, b0.x);
                        fma2(acc[r][1], xx, b0.y);
                        fma2(acc[r][2], xx, b1.x);
                        fma2(acc[r][3], xx, b1.y);
                    }
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            const int row = r * kRowGroups + rg;
            if (row >= w.rows) continue;
            float* o = (MODE == F32_TILE || MODE == F32_L2L ? a.L : a.out) + (int64_t)(w.row0 + row) * a.ld;
            // columns P .. ld - 1: zeros (zero operator columns) or NaN, read by nothing
            if (n0 < a.ld) {
                float4 v;
                unpack2(acc[r][0], v.x, v.y);
                unpack2(acc[r][1], v.z, v.w);
                *reinterpret_cast<float4*>(o + n0) = v;
            }
            if (n1 < a.ld) {
                float4 v;
                unpack2(acc[r][2], v.x, v.y);
                unpack2(acc[r][3], v.z, v.w);
                *reinterpret_cast<float4*>(o + n1) = v;
            }
        }
    }
    asm volatile("cp.async.wait_all;" ::: "memory");
}

// operators transposed and padded: [op][kch * 32][split][nc], zero beyond P
__global__ void k_f32_pack(int op0, int nops, int P, int kpad, int ntot, int transposed,
                           const float* __restrict__ T, float* ops) {
    const int64_t per = (int64_t)kpad * ntot;
    for (int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; e < nops * per;
         e += (int64_t)gridDim.x * blockDim.x) {
        const int o = (int)(e / per), k = (int)(e % per / ntot), n = (int)(e % ntot);
        float v = 0.f;
        if (k < P && n < P)
            v = T[(int64_t)o * P * P + (transposed ? (int64_t)k * P + n : (int64_t)n * P + k)];
        ops[(int64_t)(op0 + o) * per + e % per] = v;
    }
}

F32Args f32_args(const Workspace& ws) {
    F32Args a;
    memset(&a, 0, sizeof a);
    const F32Cols c = f32_cols(ws.P);
    a.P = ws.P;
    a.ld = ws.ld;
    a.kch = (ws.P + 31) / 32;
    a.nc = c.nc;
    a.split = c.split;
    a.op_vals = (int64_t)a.kch * 32 * c.split * c.nc;
    a.ops = (const float*)ws.T_f32;
    a.linfo = ws.linfo;
    a.code = ws.code;
    a.cid = ws.cid;
    a.M = (const float*)ws.M;
    a.L = (float*)ws.L;
    return a;
}

template <int R>
int f32_smem_bytes(const F32Args& a) {
    return kF32Stages * (kRowGroups * R * kAStride + 32 * a.nc) * (int)sizeof(float);
}

template <int MODE, int R>
cudaError_t f32_launch(const F32Args& a, int64_t units, const Workspace& ws, cudaStream_t s) {
    // blocks per SM by shared memory and threads
    const int smem = f32_smem_bytes<R>(a), thr = kRowGroups * a.nc / 8;
    const int per = std::max(1, std::min(std::min(220 * 1024 / (smem + 4096), 2048 / thr), 4));
    const int64_t grid = std::max<int64_t>(1, std::min<int64_t>(units * a.split, (int64_t)ws.sms * per));
    return launch_pdl(k_f32_gemm<MODE, R>, dim3((unsigned)grid), dim3((unsigned)thr), (size_t)smem, s, a);
}
// 128-row tiles when they fill the GPU, else 32-row tiles
template <int MODE>
cudaError_t f32_rows(const F32Args& a, int64_t rows, const Workspace& ws, cudaStream_t s) {
    const int64_t t128 = rows / 128 + 8;
    if (t128 >= 2 * ws.sms) return f32_launch<MODE, 8>(a, t128, ws, s);
    return f32_launch<MODE, 2>(a, rows / 32 + 8, ws, s);
}

}  // namespace

size_t m2l_f32_operator_bytes(int p) {
    const int P = (p + 1) * (p + 1);
    const F32Cols c = f32_cols(P);
    return sizeof(float) * (size_t)kF32Ops * ((P + 31) / 32 * 32) * (c.split * c.nc);
}

cudaError_t m2l_f32_init() {
    int16_t off[8][189];
    host_m2l_offsets(off);
    cudaError_t e = cudaMemcpyToSymbol(c_f32_off, off, sizeof off);
    for (const void* f : {(const void*)k_f32_gemm<F32_PAIR, 8>, (const void*)k_f32_gemm<F32_TILE, 8>,
                          (const void*)k_f32_gemm<F32_TILE, 2>, (const void*)k_f32_gemm<F32_M2M, 8>,
                          (const void*)k_f32_gemm<F32_M2M, 2>, (const void*)k_f32_gemm<F32_L2L, 8>,
                          (const void*)k_f32_gemm<F32_L2L, 2>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
    return e;
}

cudaError_t m2l_f32_pack(const Workspace& ws) {
    const F32Args a = f32_args(ws);
    struct Set {
        int op0, n, tr;
        const void* T;
    };
    for (const Set& s : {Set{0, 343, 0, ws.T_m2l}, Set{kF32M2M, 8, 1, ws.T_m2m},
                         Set{kF32L2L, 8, 0, ws.T_l2l}}) {
        k_f32_pack<<<152 * 8, 256>>>(s.op0, s.n, a.P, a.kch * 32, a.split * a.nc, s.tr,
                                     (const float*)s.T, (float*)ws.T_f32);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    return cudaStreamSynchronize(0);
}

cudaError_t launch_f32_pairs(Workspace& ws, cudaStream_t s) {
    const PairList L = pair_list(ws);
    F32Args a = f32_args(ws);
    a.hdr = L.hdr;
    a.items = L.items;
    a.pairs = L.pairs;
    a.out = (float*)ws.pp_part;
    return f32_launch<F32_PAIR, 8>(a, ws.pp_item_cap, ws, s);
}

cudaError_t launch_f32_tiles(int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    const DenseLayout dl = dense_layout(D);
    F32Args a = f32_args(ws);
    a.level = l;
    a.off_level = dl.off[l];
    a.off_other = l >= 3 ? dl.off[l - 1] : 0;
    return f32_rows<F32_TILE>(a, level_cap(n, l), ws, s);
}

cudaError_t launch_f32_m2m(int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    F32Args a = f32_args(ws);
    a.level = l;
    a.off_other = dense_layout(D).off[l + 1];
    a.out = (float*)ws.M;
    return f32_rows<F32_M2M>(a, level_cap(n, l), ws, s);
}

cudaError_t launch_f32_l2l(int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    F32Args a = f32_args(ws);
    a.level = l;
    a.off_other = dense_layout(D).off[l - 1];
    return f32_rows<F32_L2L>(a, level_cap(n, l), ws, s);
}

}  // namespace pt
