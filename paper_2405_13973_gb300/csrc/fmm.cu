// fmm.cu -- the FMM stages on the CUDA cores (Sec. 2.3.2) and the order of
// one evaluation's launches (run_fmm: main chain and side stream).
//
// Upward pass: P2M at the leaves (Eq. FMM_coul2; on the tensor-core path
// also at the leaves' parents, straight from their ions), M2M to the parents.
// Downward pass: at every level l >= 2 the local expansion of a cell is the
// L2L shift of its parent's plus the M2L conversion (Eq. FMM_local) of the
// multipole expansions of the 189 cells that are children of the parent's
// neighbours but not neighbours themselves.  At the leaves the far field is
// the gradient of the local expansion (L2P) and the near field the direct sum
// over the 27 adjacent leaves (P2P).
//
// Cells of one level are stored octant-major, so a tile of target cells
// shares its octant and therefore the same 189 source offsets: M2L becomes,
// per offset o, a dense product L[:, tile] += T_o * M[:, src(tile, o)], the
// L2L shift being one more such product with the parent's L.
//
// Everything is templated on the arithmetic type (double: PT_FP64, float:
// PT_FP32 and the CUDA-core stages of PT_MIXED_TF32X3).  Coefficients are in
// the normalised real storage of harmonics.cuh, scaled by the cell size.
#include <cuda_runtime.h>

#include "bf16split.cuh"
#include "fmm_math.cuh"
#include "harmonics.cuh"
#include "internal.h"
#include "join.cuh"

namespace pt {

__constant__ HarmTables<double> c_tab_d;
__constant__ HarmTables<float> c_tab_f;
// the same tables in global memory, for kernels whose lanes read them at
// different m (constant memory would serialise those reads)
__device__ HarmTables<double> g_tab_d;
__device__ HarmTables<float> g_tab_f;
// M2L source offsets per target octant: packed (ox+3)*49 + (oy+3)*7 + (oz+3),
// o = target - source, o_a in [b_a - 3, b_a + 2] with b the octant bits,
// excluding the 27 neighbours.
__constant__ int16_t c_m2l_off[8][189];

template <typename T>
__device__ __forceinline__ const HarmTables<T>& tab();
template <>
__device__ __forceinline__ const HarmTables<double>& tab<double>() { return c_tab_d; }
template <>
__device__ __forceinline__ const HarmTables<float>& tab<float>() { return c_tab_f; }
template <typename T>
__device__ __forceinline__ const HarmTables<T>& gtab();
template <>
__device__ __forceinline__ const HarmTables<double>& gtab<double>() { return g_tab_d; }
template <>
__device__ __forceinline__ const HarmTables<float>& gtab<float>() { return g_tab_f; }

void host_m2l_offsets(int16_t out[8][189]) {
    for (int oct = 0; oct < 8; ++oct) {
        int b[3] = {(oct >> 2) & 1, (oct >> 1) & 1, oct & 1};
        int k = 0;
        for (int ox = b[0] - 3; ox <= b[0] + 2; ++ox)
            for (int oy = b[1] - 3; oy <= b[1] + 2; ++oy)
                for (int oz = b[2] - 3; oz <= b[2] + 2; ++oz) {
                    if (ox >= -1 && ox <= 1 && oy >= -1 && oy <= 1 && oz >= -1 && oz <= 1) continue;
                    out[oct][k++] = (int16_t)((ox + 3) * 49 + (oy + 3) * 7 + (oz + 3));
                }
    }
}


// Sorted ion records (written by the tree build): the FP64 path keeps
// (u, q) in double; the FP32 paths keep u in 30-bit fixed point and q as
// float bits (int4), so that near-field separations are exact integers.
template <typename T>
struct Ion;
template <>
struct Ion<double> {
    using rec = double4_32a;
    static __device__ __forceinline__ void get(const rec& r, double& x, double& y, double& z,
                                               double& q) {
        x = r.x; y = r.y; z = r.z; q = r.w;
    }
    // (x_t - x_s)/s for a source in the leaf at integer offset d from the target's
    static __device__ __forceinline__ void sep(const rec& t, const rec& o, int dx, int dy, int dz,
                                               double& rx, double& ry, double& rz) {
        rx = (t.x - o.x) - dx;
        ry = (t.y - o.y) - dy;
        rz = (t.z - o.z) - dz;
    }
    // a source expressed in the target leaf's frame (u + d)
    static __device__ __forceinline__ rec shifted(const rec& o, int dx, int dy, int dz) {
        return make_double4_32a(o.x + dx, o.y + dy, o.z + dz, o.w);
    }
    static __device__ __forceinline__ void sep_shifted(const rec& t, const rec& o, double& rx,
                                                       double& ry, double& rz, double& q) {
        rx = t.x - o.x;
        ry = t.y - o.y;
        rz = t.z - o.z;
        q = o.w;
    }
};
template <>
struct Ion<float> {
    using rec = int4;
    static __device__ __forceinline__ void get(const rec& r, float& x, float& y, float& z,
                                               float& q) {
        x = __int2float_rn(r.x) * 0x1p-30f;
        y = __int2float_rn(r.y) * 0x1p-30f;
        z = __int2float_rn(r.z) * 0x1p-30f;
        q = __int_as_float(r.w);
    }
    // |t - o| < 2^30 and |d| 2^30 <= 2^30: the integer difference fits in 31 bits
    static __device__ __forceinline__ void sep(const rec& t, const rec& o, int dx, int dy, int dz,
                                               float& rx, float& ry, float& rz) {
        rx = __int2float_rn((t.x - o.x) - dx * (1 << 30)) * 0x1p-30f;
        ry = __int2float_rn((t.y - o.y) - dy * (1 << 30)) * 0x1p-30f;
        rz = __int2float_rn((t.z - o.z) - dz * (1 << 30)) * 0x1p-30f;
    }
    // a source in the target leaf's frame: u + d 2^30 stays within
    // [-2^29 - 2^30, 2^29 - 1 + 2^30], so u_t - (u_s + d 2^30) fits in int32
    static __device__ __forceinline__ rec shifted(const rec& o, int dx, int dy, int dz) {
        return make_int4(o.x + dx * (1 << 30), o.y + dy * (1 << 30), o.z + dz * (1 << 30), o.w);
    }
    static __device__ __forceinline__ void sep_shifted(const rec& t, const rec& o, float& rx,
                                                       float& ry, float& rz, float& q) {
        rx = __int2float_rn(t.x - o.x) * 0x1p-30f;
        ry = __int2float_rn(t.y - o.y) * 0x1p-30f;
        rz = __int2float_rn(t.z - o.z) * 0x1p-30f;
        q = __int_as_float(o.w);
    }
};

// s + v with the rounding error carried in c (Kahan-Babuska / Neumaier).
template <typename T>
__device__ __forceinline__ void kb_add(T& s, T& c, T v) {
    T t = s + v;
    if (fabs(s) >= fabs(v)) c += (s - t) + v;
    else c += (v - t) + s;
    s = t;
}

// The same in FP64 with one instruction of the FP64 pipe less: the order by
// exponent is enough for the error to be exact.
__device__ __forceinline__ void kb_add_d(double& s, double& c, double v) {
    const double t = s + v;
    const bool ge = (__double2hiint(s) & 0x7ff00000) >= (__double2hiint(v) & 0x7ff00000);
    c += (ge ? v : s) - (t - (ge ? s : v));
    s = t;
}

// Position of a sorted ion in the frame of its ancestor s levels above its
// leaf: o = the leaf's integer position inside the ancestor (0 .. 2^s - 1
// per axis), u_anc = (u_leaf + o + 1/2 - 2^s / 2) / 2^s, in ancestor units.
__device__ __forceinline__ void ion_in_ancestor(const Ion<float>::rec& r, int s, int ox, int oy,
                                                int oz, float& x, float& y, float& z, float& q) {
    const float sc = __int_as_float((127 - 30 - s) << 23);  // 2^-(30+s)
    const int half = 1 << s;
    const long long u = 1ll << 29;  // 1/2 in 30-bit fixed point
    x = __ll2float_rn((long long)r.x + (long long)(2 * ox + 1 - half) * u) * sc;
    y = __ll2float_rn((long long)r.y + (long long)(2 * oy + 1 - half) * u) * sc;
    z = __ll2float_rn((long long)r.z + (long long)(2 * oz + 1 - half) * u) * sc;
    q = __int_as_float(r.w);
}
__device__ __forceinline__ void ion_in_ancestor(const Ion<double>::rec& r, int s, int ox, int oy,
                                                int oz, double& x, double& y, double& z, double& q) {
    const double sc = ldexp(1.0, -s), c = 0.5 - 0.5 * (double)(1 << s);
    x = (r.x + ((double)ox + c)) * sc;
    y = (r.y + ((double)oy + c)) * sc;
    z = (r.z + ((double)oz + c)) * sc;
    q = r.w;
}

constexpr int kPmax = (kMaxOrder + 1) * (kMaxOrder + 1);
constexpr int kP2mThreads = 128;
constexpr int kP2mIons = 32;

// ---------------------------------------------------------------------------
// P2M: one block per leaf.  Each thread evaluates conj(Y^_n^m(u)) q of one ion
// (all n, m, by the column recurrences) into shared memory, then each thread
// owns coefficients and sums them over the leaf's ions in slot order
// (deterministic).  Leaves with more ions than kP2mIons are done in passes.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void k_p2m_body(const BlockId& blk, int D, int p, int ld, const LevelInfo* linfo,
                                                     const int32_t* __restrict__ cstart,
                                                     const int32_t* __restrict__ ccount,
                                                     const typename Ion<T>::rec* __restrict__ sorted,
                                                     T* __restrict__ M, uint16_t* Mp) {
    extern __shared__ unsigned char p2m_smem[];
    const int P = (p + 1) * (p + 1);
    T* terms = reinterpret_cast<T*>(p2m_smem);  // [kP2mIons][P]
    const HarmTables<T>& t = tab<T>();
    const int g0 = linfo->gbase[D], g1 = linfo->gbase[D + 1];
    for (int g = g0 + (int)blk.x; g < g1; g += (int)blk.nx) {
        const int s = cstart[g], k = ccount[g];
        T acc[(kMaxOrder + 1) * (kMaxOrder + 1) / kP2mThreads + 1];
        constexpr int NA = (kMaxOrder + 1) * (kMaxOrder + 1) / kP2mThreads + 1;
#pragma unroll
        for (int r = 0; r < NA; ++r) acc[r] = T(0);
        for (int i0 = 0; i0 < k; i0 += kP2mIons) {
            const int ni = min(kP2mIons, k - i0);
            __syncthreads();
            if (threadIdx.x < ni) {
                T x, y, z, q;
                Ion<T>::get(sorted[s + i0 + threadIdx.x], x, y, z, q);
                T* row = terms + threadIdx.x * P;
                for_each_ups<T>(p, x, y, z, t, [&](int n, int m, T re, T im) {
                    const int idx = re_idx(n, m);
                    row[idx] = q * re;
                    if (m > 0) row[idx + 1] = -q * im;
                });
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < NA; ++r) {
                const int c = threadIdx.x + r * kP2mThreads;
                if (c < P)
                    for (int i = 0; i < ni; ++i) acc[r] += terms[i * P + c];
            }
        }
#pragma unroll
        for (int r = 0; r < NA; ++r) {
            const int c = threadIdx.x + r * kP2mThreads;
            if (c < P) {
                M[(int64_t)g * ld + c] = acc[r];
                if (Mp) store_pieces(Mp, g, ld, c, (float)acc[r]);  // BF16x3 operand
            }
        }
    }
}
template <typename T>
__global__ void __launch_bounds__(kP2mThreads) k_p2m(int D, int p, int ld, const LevelInfo* linfo,
                                                     const int32_t* __restrict__ cstart,
                                                     const int32_t* __restrict__ ccount,
                                                     const typename Ion<T>::rec* __restrict__ sorted,
                                                     T* __restrict__ M, uint16_t* Mp) {
    k_p2m_body<T>(solo_block(), D, p, ld, linfo, cstart, ccount, sorted, M, Mp);
}

// ---------------------------------------------------------------------------
// P2M and L2P in FP64.  The FP64 units serve two lanes a clock, and a warp
// instruction occupies them as long with seven live lanes as with 32, so the
// lanes hold the ions of several leaves: a block takes the leaves that begin
// in its window of kSlotWindow sorted slots, and a thread evaluates all
// (p + 1)^2 harmonics of one ion (tables from constant memory, every lane at
// the same (n, m)).  With a block per leaf (5 to 10 ions), P2M kept 7 of 32
// lanes busy, and L2P spent its lanes on recurrences shared by eight of them.
// ---------------------------------------------------------------------------
constexpr int kSlotThreads = 64, kSlotWindow = 48;
// below these ion counts a thread per ion leaves most of the FP64 units idle
// and its chain of recurrences is the time, so a block per leaf is faster
// (P2M, p = 8 / 12: 8,000 ions 44 / 71 us by windows, 32 / 64 by leaves,
// 16,000 ions 46 / 82 and 69 / 136; L2P: 4,000 ions 46 / 91 and 44 / 62, 8,000
// ions 45 / 89 and 73 / 100)
constexpr int64_t kP2mSlotIons = 10240, kL2pSlotIons = 7168;
// FP32 (p <= 15): ions from which k_l2p_f32 takes one thread an ion instead of
// four (us, k_l2p / 4 threads / 1 thread): 300 ions (p = 12) 11 / 9.7 / -,
// 1,500 16.5 / 12.8 / -, 5,000 26 / 20 / 39, 10,000 31 / 21 / 32, 23,000
// (p = 8) 41 / 34 / 22, 30,000 (p = 3) 21 / 20 / 12, 1e5 (p = 12)
// 220 / 158 / 115.  Members of an ensemble share a launch and fill the chip
// together: one thread (256 crystals, k_l2p / 1 thread: 1,700 / 726 us).
constexpr int64_t kL2pF32Ions = 16384;

// the slots [s0, s1) of the leaves that begin in window b; false if none does
__device__ __forceinline__ bool slot_window(int64_t n, int b, const int32_t* __restrict__ leaf_of,
                                            const int32_t* __restrict__ cstart,
                                            const int32_t* __restrict__ ccount, int& s0, int& s1,
                                            int window = kSlotWindow) {
    const int w0 = b * window, w1 = (int)min(n, (int64_t)w0 + window);
    const int gf = leaf_of[w0], gl = leaf_of[w1 - 1];
    s0 = cstart[gf];
    if (s0 < w0) s0 += ccount[gf];
    s1 = cstart[gl] + ccount[gl];
    return s0 < w1;
}

// row stride of one ion's terms: odd, so that a column of rows has no bank conflicts
__host__ __device__ inline int p2m_f64_stride(int P) { return P | 1; }

__global__ void __launch_bounds__(kSlotThreads) k_p2m_f64(
    int64_t n, int p, int ld, const int32_t* __restrict__ leaf_of,
    const int32_t* __restrict__ cstart, const int32_t* __restrict__ ccount,
    const Ion<double>::rec* __restrict__ sorted, double* __restrict__ M) {
    extern __shared__ double slot_smem[];  // [kSlotThreads][stride]
    __shared__ int s_leaf[kSlotThreads + 1];
    const int P = (p + 1) * (p + 1), S = p2m_f64_stride(P), tid = threadIdx.x;
    pdl_wait();
    int s0, s1;
    if (!slot_window(n, blockIdx.x, leaf_of, cstart, ccount, s0, s1)) return;  // uniform
    constexpr int NA = (kPmax + kSlotThreads - 1) / kSlotThreads;
    double acc[NA];
#pragma unroll
    for (int r = 0; r < NA; ++r) acc[r] = 0.0;
    for (int p0 = s0; p0 < s1; p0 += kSlotThreads) {
        const int ni = min(kSlotThreads, s1 - p0);
        __syncthreads();
        if (tid < ni) {
            s_leaf[tid] = leaf_of[p0 + tid];
            double x, y, z, q;
            Ion<double>::get(sorted[p0 + tid], x, y, z, q);
            double* row = slot_smem + tid * S;
            for_each_ups<double>(p, x, y, z, c_tab_d, [&](int nn, int m, double re, double im) {
                const int idx = re_idx(nn, m);
                row[idx] = q * re;
                if (m > 0) row[idx + 1] = -q * im;
            });
        }
        if (tid == 0) s_leaf[ni] = p0 + ni < s1 ? leaf_of[p0 + ni] : -1;
        __syncthreads();
        // each thread its coefficients, ion after ion; a leaf ends where the
        // next slot belongs to another
        for (int i = 0; i < ni; ++i) {
#pragma unroll
            for (int r = 0; r < NA; ++r) {
                const int c = tid + r * kSlotThreads;
                if (c < P) acc[r] += slot_smem[i * S + c];
            }
            const int g = s_leaf[i];
            if (s_leaf[i + 1] != g) {
#pragma unroll
                for (int r = 0; r < NA; ++r) {
                    const int c = tid + r * kSlotThreads;
                    if (c < P) M[(int64_t)g * ld + c] = acc[r];
                    acc[r] = 0.0;
                }
            }
        }
    }
}

// ---------------------------------------------------------------------------
// Direct ancestor multipoles (PT_EXPAND_DIRECT): P2M of every ion about each
// of its cells at levels lmin..D, one block per cell, as k_p2m but with u in
// the cell's frame and units and compensated sums (an ancestor's
// coefficients sum thousands of terms of both signs).  A cell's ions are the
// contiguous slots of its leaves.  Equal to P2M at the leaves followed by the
// M2M shifts, which shift a truncated expansion exactly.
// ---------------------------------------------------------------------------
constexpr int kP2mAncIons = 64;

template <typename T>
__device__ __forceinline__ void k_p2m_anc_body(
    const BlockId& blk, int D, int lmin, int p, int ld, const LevelInfo* linfo,
    const uint32_t* __restrict__ code,
    const int32_t* __restrict__ leaf_start, const int32_t* __restrict__ leaf_of,
    const typename Ion<T>::rec* __restrict__ sorted, T* __restrict__ M, uint16_t* Mp) {
    extern __shared__ unsigned char p2m_smem[];
    const int P = (p + 1) * (p + 1);
    pdl_wait();
    T* terms = reinterpret_cast<T*>(p2m_smem);  // [kP2mAncIons][P]
    const HarmTables<T>& t = tab<T>();
    const int g0 = linfo->gbase[lmin], g1 = linfo->gbase[D + 1];
    for (int g = g0 + (int)blk.x; g < g1; g += (int)blk.nx) {
        int l = lmin;
        while (l < D && g >= linfo->gbase[l + 1]) ++l;
        const int sh = D - l, mask = (1 << sh) - 1;
        const uint32_t c = code[g];
        const int s = leaf_start[(int64_t)c << (3 * sh)];
        const int k = leaf_start[((int64_t)c + 1) << (3 * sh)] - s;
        constexpr int NA = (kMaxOrder + 1) * (kMaxOrder + 1) / kP2mThreads + 1;
        T acc[NA], cmp[NA];
#pragma unroll
        for (int r = 0; r < NA; ++r) acc[r] = cmp[r] = T(0);
        for (int i0 = 0; i0 < k; i0 += kP2mAncIons) {
            const int ni = min(kP2mAncIons, k - i0);
            __syncthreads();
            if (threadIdx.x < ni) {
                T x, y, z, q;
                const int slot = s + i0 + threadIdx.x;
                int ix, iy, iz;
                demorton3(code[leaf_of[slot]], ix, iy, iz);
                ion_in_ancestor(sorted[slot], sh, ix & mask, iy & mask, iz & mask, x, y, z, q);
                T* row = terms + threadIdx.x * P;
                for_each_ups<T>(p, x, y, z, t, [&](int n, int m, T re, T im) {
                    const int idx = re_idx(n, m);
                    row[idx] = q * re;
                    if (m > 0) row[idx + 1] = -q * im;
                });
            }
            __syncthreads();
#pragma unroll
            for (int r = 0; r < NA; ++r) {
                const int cc = threadIdx.x + r * kP2mThreads;
                if (cc < P)
                    for (int i = 0; i < ni; ++i) kb_add(acc[r], cmp[r], terms[i * P + cc]);
            }
        }
#pragma unroll
        for (int r = 0; r < NA; ++r) {
            const int cc = threadIdx.x + r * kP2mThreads;
            if (cc < P) {
                const T v = acc[r] + cmp[r];
                M[(int64_t)g * ld + cc] = v;
                if (Mp) store_pieces(Mp, g, ld, cc, (float)v);  // BF16x3 operand
            }
        }
    }
}
template <typename T>
__global__ void __launch_bounds__(kP2mThreads) k_p2m_anc(
    int D, int lmin, int p, int ld, const LevelInfo* linfo, const uint32_t* __restrict__ code,
    const int32_t* __restrict__ leaf_start, const int32_t* __restrict__ leaf_of,
    const typename Ion<T>::rec* __restrict__ sorted, T* __restrict__ M, uint16_t* Mp) {
    k_p2m_anc_body<T>(solo_block(), D, lmin, p, ld, linfo, code, leaf_start, leaf_of, sorted, M, Mp);
}

// ---------------------------------------------------------------------------
// M2M: one warp per parent; lanes over output coefficients.
//   Tt: [8][P][P] transposed (in-major) so that lanes read consecutively.
// ---------------------------------------------------------------------------
template <typename T>
__global__ void __launch_bounds__(128) k_m2m(int l, int P, int ld, const LevelInfo* linfo,
                                             const uint32_t* __restrict__ code,
                                             const int32_t* __restrict__ cid, int64_t off_child,
                                             const T* __restrict__ Tt, T* M) {
    extern __shared__ unsigned char smem_raw[];
    T* sM = reinterpret_cast<T*>(smem_raw) + (threadIdx.x >> 5) * P;
    const int lane = threadIdx.x & 31;
    const int warps = (gridDim.x * blockDim.x) >> 5;
    const int g0 = linfo->gbase[l], g1 = linfo->gbase[l + 1];
    constexpr int R = ((kMaxOrder + 1) * (kMaxOrder + 1) + 31) / 32;
    for (int g = g0 + ((blockIdx.x * blockDim.x + threadIdx.x) >> 5); g < g1; g += warps) {
        const uint32_t c = code[g];
        T acc[R];
#pragma unroll
        for (int r = 0; r < R; ++r) acc[r] = T(0);
        for (int o = 0; o < 8; ++o) {
            const int gc = cid[off_child + ((c << 3) | o)];
            if (gc < 0) continue;
            __syncwarp();
            for (int k = lane; k < P; k += 32) sM[k] = M[(int64_t)gc * ld + k];
            __syncwarp();
            const T* To = Tt + (int64_t)o * P * P;
            for (int k = 0; k < P; ++k) {
                const T mk = sM[k];
#pragma unroll
                for (int r = 0; r < R; ++r) {
                    int row = lane + 32 * r;
                    if (row < P) acc[r] += To[(int64_t)k * P + row] * mk;
                }
            }
        }
#pragma unroll
        for (int r = 0; r < R; ++r) {
            int row = lane + 32 * r;
            if (row < P) M[(int64_t)g * ld + row] = acc[r];
        }
    }
}

// ---------------------------------------------------------------------------
// M2M and L2L of the small upper levels on the tensor-core paths, on the CUDA
// cores: out[g][r] (+)= sum_t Op[r][t] x_g[t], with
//   M2M (MODE 0): x_g = the M of parent g's eight children side by side
//                 (t = o P + c; absent children zero), Op = [T_0 ... T_7];
//   L2L (MODE 1): x_g = the L of child g's parent, Op = T_octant(g), added
//                 to the child's own M2L sum already in L.
// A level of a few dozen or hundred cells is latency work: a launch of the
// persistent tensor-core kernel (TMEM and barrier set-up, operator copies
// from DRAM, one partial per octant and a reduction for M2M) costs more than
// the products.  A block holds rows r0 .. r0 + 15 of the operator in shared
// memory (staged before the programmatic wait: operators are constants) and
// applies them to runs of kShCells cells; warp w owns rows w and w + 8, its
// lanes split the dot products and a butterfly sums them (every lane gets the
// same value: the order is fixed, results are deterministic).
// ---------------------------------------------------------------------------
constexpr int kShRows = 16;
constexpr int kShThreads = 256;
template <int MODE>
struct ShCells { static constexpr int v = MODE == 0 ? 8 : 16; };

// 4-byte asynchronous copy global -> shared (zero-filled when !valid): the
// staging loops issue every copy before waiting once
__device__ __forceinline__ void cp_async4(void* dst, const void* src, bool valid) {
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src),
                 "r"(valid ? 4 : 0)
                 : "memory");
}
__device__ __forceinline__ void cp_async_wait_all() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// row stride of the staged operator: K rounded up to 2 mod 32 (the M2M
// staging writes two values of t for 16 rows per warp without conflicts)
__host__ __device__ inline int sh_stride(int K) { return K + ((2 - K % 32) % 32 + 32) % 32; }

template <typename T, int MODE>
size_t shift_rows_smem(int P) {
    const int K = MODE == 0 ? 8 * P : P;
    return (size_t)(kShRows * sh_stride(K) + ShCells<MODE>::v * K) * sizeof(T);
}

template <typename T, int MODE>
__device__ __forceinline__ void k_shift_rows_body(const BlockId& blk, int l, int P, int ld,
                                                           const LevelInfo* linfo,
                                                           const uint32_t* __restrict__ code,
                                                           const int32_t* __restrict__ cid,
                                                           int64_t off_nb,
                                                           const T* __restrict__ Op, T* Y,
                                                           uint16_t* Mp) {
    static_assert(sizeof(T) == 4, "FP32 plans only (4-byte asynchronous copies)");
    constexpr int CG = ShCells<MODE>::v;
    extern __shared__ unsigned char smem_raw[];
    __shared__ int s_src[CG * (MODE == 0 ? 8 : 1)];
    const int K = MODE == 0 ? 8 * P : P, S = sh_stride(K);
    T* sOp = reinterpret_cast<T*>(smem_raw);  // [kShRows][S]
    T* sX = sOp + kShRows * S;                // [CG][K]
    const int tid = threadIdx.x, w = tid >> 5, lane = tid & 31;
    const int r0 = (int)blk.x * kShRows;
    const int oct = MODE == 1 ? (int)blk.y : 0;
    if (MODE == 0) {
        // Op = T_m2m transposed, [o][c][r]: element (r, t = o P + c) at t P + r
        for (int e = tid; e < K * kShRows; e += kShThreads) {
            const int t = e >> 4, rr = e & 15, r = r0 + rr;
            cp_async4(&sOp[rr * S + t], Op + (int64_t)t * P + (r < P ? r : 0), r < P);
        }
    } else {
        const T* To = Op + (int64_t)oct * P * P;  // T_l2l row-major [o][r][c]
        for (int rr = w; rr < kShRows; rr += kShThreads / 32) {
            const int r = r0 + rr;
            for (int c = lane; c < K; c += 32)
                cp_async4(&sOp[rr * S + c], To + (int64_t)(r < P ? r : 0) * P + c, r < P);
        }
    }
    pdl_wait();
    int g0, g1;
    if (MODE == 0) {
        g0 = linfo->gbase[l];
        g1 = linfo->gbase[l + 1];
    } else {
        g0 = linfo->oct_start[l][oct];
        g1 = linfo->oct_start[l][oct + 1];
    }
    const int nch = (g1 - g0 + CG - 1) / CG;
    const int ch0 = MODE == 0 ? (int)blk.y : (int)blk.z;
    const int chs = MODE == 0 ? (int)blk.ny : (int)blk.nz;
    const T* op0 = sOp + w * S;
    const T* op1 = sOp + (w + 8) * S;
    for (int ch = ch0; ch < nch; ch += chs) {
        const int gb = g0 + ch * CG, nc = min(CG, g1 - gb);
        __syncthreads();  // the previous run is done with sX and s_src
        if (MODE == 0) {
            if (tid < CG * 8) {
                const int ci = tid >> 3, o = tid & 7;
                s_src[tid] = ci < nc ? cid[off_nb + (((int64_t)code[gb + ci] << 3) | o)] : -1;
            }
        } else if (tid < CG) {
            s_src[tid] = tid < nc ? cid[off_nb + (code[gb + tid] >> 3)] : -1;
        }
        __syncthreads();
        // x rows: (cell, octant) of M2M, one per cell for L2L
        for (int q = w; q < CG * (MODE == 0 ? 8 : 1); q += kShThreads / 32) {
            const int src = s_src[q];
            T* dst = sX + (MODE == 0 ? (q >> 3) * K + (q & 7) * P : q * K);
            const T* from = Y + (int64_t)(src >= 0 ? src : 0) * ld;
            for (int c = lane; c < P; c += 32) cp_async4(&dst[c], from + c, src >= 0);
        }
        cp_async_wait_all();  // this thread's copies (and, first time round, the operator's)
        __syncthreads();
        T a0[CG], a1[CG];
#pragma unroll
        for (int ci = 0; ci < CG; ++ci) a0[ci] = a1[ci] = T(0);
        for (int t = lane; t < K; t += 32) {
            const T u0 = op0[t], u1 = op1[t];
#pragma unroll
            for (int ci = 0; ci < CG; ++ci) {
                const T x = sX[ci * K + t];
                a0[ci] += u0 * x;
                a1[ci] += u1 * x;
            }
        }
        T v0 = T(0), v1 = T(0);
#pragma unroll
        for (int ci = 0; ci < CG; ++ci) {
#pragma unroll
            for (int o = 16; o >= 1; o >>= 1) {
                a0[ci] += __shfl_xor_sync(0xffffffffu, a0[ci], o);
                a1[ci] += __shfl_xor_sync(0xffffffffu, a1[ci], o);
            }
            if (lane == ci) {
                v0 = a0[ci];
                v1 = a1[ci];
            }
        }
        if (lane < nc) {  // lane ci stores cell ci's rows w and w + 8
            T* y = Y + (int64_t)(gb + lane) * ld;
            const int ra = r0 + w, rb = r0 + w + 8;
            if (MODE == 0) {
                if (ra < P) y[ra] = v0;
                if (rb < P) y[rb] = v1;
                if (Mp) {  // BF16x3 operand of the M2L
                    if (ra < P) store_pieces(Mp, gb + lane, ld, ra, (float)v0);
                    if (rb < P) store_pieces(Mp, gb + lane, ld, rb, (float)v1);
                }
            } else {
                if (ra < P) y[ra] += v0;
                if (rb < P) y[rb] += v1;
            }
        }
    }
}
template <typename T, int MODE>
__global__ void __launch_bounds__(kShThreads) k_shift_rows(int l, int P, int ld,
                                                           const LevelInfo* linfo,
                                                           const uint32_t* __restrict__ code,
                                                           const int32_t* __restrict__ cid,
                                                           int64_t off_nb,
                                                           const T* __restrict__ Op, T* Y,
                                                           uint16_t* Mp) {
    k_shift_rows_body<T, MODE>(solo_block(), l, P, ld, linfo, code, cid, off_nb, Op, Y, Mp);
}

// ---------------------------------------------------------------------------
// M2L (+ folded L2L) on the CUDA cores: block = 64 output rows x 32 targets of
// one octant; loops over the 189 offsets (and the parent shift), each a
// 64 x P x 32 product staged through shared memory.
// ---------------------------------------------------------------------------
constexpr int kRT = 64, kNT = 32, kKC = 16;

template <typename T>
__global__ void __launch_bounds__(256) k_m2l_simt(int l, int P, int ld, const LevelInfo* linfo,
                                                  const uint32_t* __restrict__ code,
                                                  const int32_t* __restrict__ cid, int64_t off_l,
                                                  int64_t off_parent, const T* __restrict__ M,
                                                  T* L, const T* __restrict__ Tm2l,
                                                  const T* __restrict__ Tl2l) {
    __shared__ T As[kKC][kRT];
    __shared__ T Bs[kKC][kNT];
    __shared__ const T* src[kNT];
    __shared__ int tile_oct, tile_base, tile_n;
    __shared__ int s_oct[9];
    const int tid = threadIdx.x;
    if (tid < 9) s_oct[tid] = linfo->oct_start[l][tid];
    __syncthreads();
    if (tid == 0) {
        int b = blockIdx.x, acc = 0;
        tile_n = 0;
        for (int o = 0; o < 8; ++o) {
            int s0 = s_oct[o], s1 = s_oct[o + 1];
            int nt = (s1 - s0 + kNT - 1) / kNT;
            if (b < acc + nt) {
                tile_oct = o;
                tile_base = s0 + (b - acc) * kNT;
                tile_n = min(kNT, s1 - tile_base);
                break;
            }
            acc += nt;
        }
    }
    __syncthreads();
    if (tile_n <= 0) return;
    const int oct = tile_oct, base = tile_base, ntile = tile_n;
    const int row0 = blockIdx.y * kRT;
    const int ty = tid >> 4, tx = tid & 15;
    const int lim = 1 << l;
    T acc[4][2];
#pragma unroll
    for (int i = 0; i < 4; ++i) acc[i][0] = acc[i][1] = T(0);
    const int nterms = 189 + (l >= 3 ? 1 : 0);
    for (int term = 0; term < nterms; ++term) {
        const T* A;
        if (term < 189) {
            const int opi = c_m2l_off[oct][term];
            A = Tm2l + (int64_t)opi * P * P;
            if (tid < kNT) {
                const T* sp = nullptr;
                if (tid < ntile) {
                    int ix, iy, iz;
                    demorton3(code[base + tid], ix, iy, iz);
                    int sx = ix - (opi / 49 - 3), sy = iy - ((opi / 7) % 7 - 3),
                        sz = iz - (opi % 7 - 3);
                    if (sx >= 0 && sx < lim && sy >= 0 && sy < lim && sz >= 0 && sz < lim) {
                        int gs = cid[off_l + morton3(sx, sy, sz)];
                        if (gs >= 0) sp = M + (int64_t)gs * ld;
                    }
                }
                src[tid] = sp;
            }
        } else {
            A = Tl2l + (int64_t)oct * P * P;
            if (tid < kNT) {
                const T* sp = nullptr;
                if (tid < ntile) {
                    int gp = cid[off_parent + (code[base + tid] >> 3)];
                    if (gp >= 0) sp = L + (int64_t)gp * ld;
                }
                src[tid] = sp;
            }
        }
        int any = __syncthreads_or(tid < kNT && src[tid] != nullptr);
        if (!any) continue;
        for (int k0 = 0; k0 < P; k0 += kKC) {
#pragma unroll
            for (int e = 0; e < (kRT * kKC) / 256; ++e) {
                int idx = tid + 256 * e;
                int r = idx / kKC, kk = idx % kKC;
                int row = row0 + r, col = k0 + kk;
                As[kk][r] = (row < P && col < P) ? A[(int64_t)row * P + col] : T(0);
            }
#pragma unroll
            for (int e = 0; e < (kNT * kKC) / 256; ++e) {
                int idx = tid + 256 * e;
                int j = idx / kKC, kk = idx % kKC;
                const T* sp = src[j];
                Bs[kk][j] = (sp != nullptr && k0 + kk < P) ? sp[k0 + kk] : T(0);
            }
            __syncthreads();
#pragma unroll
            for (int kk = 0; kk < kKC; ++kk) {
                T a0 = As[kk][ty * 4 + 0], a1 = As[kk][ty * 4 + 1], a2 = As[kk][ty * 4 + 2],
                  a3 = As[kk][ty * 4 + 3];
                T b0 = Bs[kk][tx * 2 + 0], b1 = Bs[kk][tx * 2 + 1];
                acc[0][0] += a0 * b0; acc[0][1] += a0 * b1;
                acc[1][0] += a1 * b0; acc[1][1] += a1 * b1;
                acc[2][0] += a2 * b0; acc[2][1] += a2 * b1;
                acc[3][0] += a3 * b0; acc[3][1] += a3 * b1;
            }
            __syncthreads();
        }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int jj = 0; jj < 2; ++jj) {
            int row = row0 + ty * 4 + i, j = tx * 2 + jj;
            if (row < P && j < ntile) L[(int64_t)(base + j) * ld + row] = acc[i][jj];
        }
}

// ---------------------------------------------------------------------------
// L2P + P2P, one thread per sorted ion; the result is written in the
// original ion order, scaled to SI (k_e / s^2 for E, k_e / s for phi, with s
// the leaf side).
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ T inv_sqrt(T r2);
template <>
__device__ __forceinline__ float inv_sqrt<float>(float r2) {
    float y = rsqrtf(r2);
    return y * (1.5f - 0.5f * r2 * y * y);  // one Newton step
}
template <>
__device__ __forceinline__ double inv_sqrt<double>(double r2) {
    return 1.0 / sqrt(r2);
}


// P2P, one block per target leaf: the sources of the 27 adjacent leaves are
// staged in shared memory in the target leaf's frame; thread (target i,
// chunk c) sums every nchunk-th source; the chunk partials are combined in a
// fixed order with compensated sums (deterministic) into near[slot] =
// (E_x, E_y, E_z, phi) in leaf units (k_e = 1, leaf side = 1).
constexpr int kNfThreads = 128;
constexpr int kNfSrc = 1024;   // staged sources per pass

__device__ __forceinline__ void k_p2p_body(
    const BlockId& blk, int D, const LevelInfo* linfo, const Ion<float>::rec* __restrict__ sorted,
    const uint32_t* __restrict__ code, const int32_t* __restrict__ cid_leaf,
    const int32_t* __restrict__ cstart, const int32_t* __restrict__ ccount, float* __restrict__ near) {
    using R = Ion<float>::rec;
    __shared__ R src[kNfSrc];
    __shared__ int nb_start[27], nb_count[27], nb_pre[28];
    __shared__ float part[kNfThreads][4];
    const int tid = threadIdx.x;
    const int lim = 1 << D;
    const int g0 = linfo->gbase[D], g1 = linfo->gbase[D + 1];
    for (int g = g0 + (int)blk.x; g < g1; g += (int)blk.nx) {
        const int ts = cstart[g], nt = ccount[g];
        int ix, iy, iz;
        demorton3(code[g], ix, iy, iz);
        if (tid < 27) {
            const int dx = tid / 9 - 1, dy = (tid / 3) % 3 - 1, dz = tid % 3 - 1;
            const int nx = ix + dx, ny = iy + dy, nz = iz + dz;
            int st = 0, ct = 0;
            if (nx >= 0 && ny >= 0 && nz >= 0 && nx < lim && ny < lim && nz < lim) {
                const int gn = cid_leaf[morton3(nx, ny, nz)];
                if (gn >= 0) {
                    st = cstart[gn];
                    ct = ccount[gn];
                }
            }
            nb_start[tid] = st;
            nb_count[tid] = ct;
        }
        __syncthreads();
        if (tid == 0) {
            int acc = 0;
            for (int k = 0; k < 27; ++k) {
                nb_pre[k] = acc;
                acc += nb_count[k];
            }
            nb_pre[27] = acc;
        }
        __syncthreads();
        const int ns = nb_pre[27];
        for (int t0 = 0; t0 < nt; t0 += kNfThreads) {   // targets in blocks of 128
            const int ntb = min(kNfThreads, nt - t0);
            const int nch = kNfThreads / ntb;            // source chunks per target
            const int ti = tid % ntb, ch = tid / ntb;
            const bool active = ch < nch;
            const R me = sorted[ts + t0 + ti];
            float ex = 0, ey = 0, ez = 0, ph = 0, cex = 0, cey = 0, cez = 0, cph = 0;
            for (int s0 = 0; s0 < ns; s0 += kNfSrc) {    // sources in passes of kNfSrc
                const int nsb = min(kNfSrc, ns - s0);
                __syncthreads();
                for (int j = tid; j < nsb; j += kNfThreads) {
                    const int v = s0 + j;
                    int k = 0;  // largest k with nb_pre[k] <= v (binary search over 28 bounds)
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (k + step <= 26 && nb_pre[k + step] <= v) k += step;
                    const int dx = k / 9 - 1, dy = (k / 3) % 3 - 1, dz = k % 3 - 1;
                    const int slot = nb_start[k] + (v - nb_pre[k]);
                    src[j] = Ion<float>::shifted(sorted[slot], dx, dy, dz);
                }
                __syncthreads();
                if (active) {
                    // the target's own entry: leaf offset d = 0 is neighbour 13
                    const int self = nb_pre[13] + (t0 + ti) - s0;
                    // plain sums over blocks of 64 sources, compensated across blocks
                    for (int jb = ch; jb < nsb; jb += 64 * nch) {
                        const int je = min(nsb, jb + 64 * nch);
                        float px = 0, py = 0, pz = 0, pp = 0;
                        for (int j = jb; j < je; j += nch) {
                            if (j == self) continue;
                            float rx, ry, rz, q;
                            Ion<float>::sep_shifted(me, src[j], rx, ry, rz, q);
                            const float r2 = rx * rx + ry * ry + rz * rz;
                            const float ir = inv_sqrt<float>(r2);
                            const float qi = q * ir;
                            const float q3 = qi * ir * ir;
                            px += q3 * rx;
                            py += q3 * ry;
                            pz += q3 * rz;
                            pp += qi;
                        }
                        kb_add(ex, cex, px);
                        kb_add(ey, cey, py);
                        kb_add(ez, cez, pz);
                        kb_add(ph, cph, pp);
                    }
                }
            }
            part[tid][0] = ex + cex;
            part[tid][1] = ey + cey;
            part[tid][2] = ez + cez;
            part[tid][3] = ph + cph;
            __syncthreads();
            if (tid < ntb) {
                // fixed-order compensated combination of the chunk partials
                float sx = 0, sy = 0, sz = 0, sp = 0, cx = 0, cy = 0, cz = 0, cp = 0;
                for (int c = 0; c < nch; ++c) {
                    const int th = c * ntb + tid;
                    kb_add(sx, cx, part[th][0]);
                    kb_add(sy, cy, part[th][1]);
                    kb_add(sz, cz, part[th][2]);
                    kb_add(sp, cp, part[th][3]);
                }
                float* o = near + 4 * (int64_t)(ts + t0 + tid);
                o[0] = sx + cx;
                o[1] = sy + cy;
                o[2] = sz + cz;
                o[3] = sp + cp;
            }
            __syncthreads();
        }
        __syncthreads();
    }
}
__global__ void __launch_bounds__(kNfThreads) k_p2p(
    int D, const LevelInfo* linfo, const Ion<float>::rec* __restrict__ sorted,
    const uint32_t* __restrict__ code, const int32_t* __restrict__ cid_leaf,
    const int32_t* __restrict__ cstart, const int32_t* __restrict__ ccount, float* __restrict__ near) {
    k_p2p_body(solo_block(), D, linfo, sorted, code, cid_leaf, cstart, ccount, near);
}

// The same in FP64.  The FP64 units serve two lanes a clock, a warp
// instruction as much as a full one, so the work is laid out for full warps:
//   * thread (target i, chunk c) as above, but the chunk partials (plain sums
//     over blocks of 64 sources, compensated across blocks: most threads have
//     one block) are added by a thread per target and component instead of a
//     thread per target, which took as long as the pair sums themselves;
//   * rsqrt (about 7 FP64 instructions) instead of a square root and a
//     division (about 25);
//   * `parts` blocks share a leaf's targets where there are few leaves, so
//     that shallow trees fill the GPU;
//   * the potential only if it is asked for.
// 1e5 sweep ions (14.5 M pairs): 2.2 ms before, 0.78 now; 1e6 ions 17.4 and
// 8.4 ms; the pair sums alone (19 instructions a pair) are 0.44 and 5.7 ms.
// (Plain adds pairwise between the chunks, without the compensation, were
// 0.12 and 0.75 ms faster.)
constexpr int kNfSrc64 = 256;  // staged sources per pass; the partials reuse their room
template <bool PHI>
__global__ void __launch_bounds__(kNfThreads, 8) k_p2p_f64(
    int D, int parts, const LevelInfo* linfo, const Ion<double>::rec* __restrict__ sorted,
    const uint32_t* __restrict__ code, const int32_t* __restrict__ cid_leaf,
    const int32_t* __restrict__ cstart, const int32_t* __restrict__ ccount,
    double* __restrict__ near) {
    using R = Ion<double>::rec;
    static_assert(kNfSrc64 >= kNfThreads, "the partials lie over the sources");
    __shared__ R src[kNfSrc64];
    __shared__ int nb_start[27], nb_pre[28];
    R* part = src;
    const int tid = threadIdx.x, lane = tid & 31;
    const int lim = 1 << D;
    const int g0 = linfo->gbase[D], units = (linfo->gbase[D + 1] - g0) * parts;
    for (int u = blockIdx.x; u < units; u += gridDim.x) {
        const int g = g0 + u / parts, ip = u % parts;
        const int nt = ccount[g], per = (nt + parts - 1) / parts;
        const int tb = min(nt, ip * per), te = min(nt, tb + per);  // this block's targets
        if (tb >= te) continue;  // uniform
        const int ts = cstart[g];
        if (tid < 32) {
            int st = 0, ct = 0;
            if (lane < 27) {
                int ix, iy, iz;
                demorton3(code[g], ix, iy, iz);
                const int nx = ix + lane / 9 - 1, ny = iy + (lane / 3) % 3 - 1, nz = iz + lane % 3 - 1;
                if (nx >= 0 && ny >= 0 && nz >= 0 && nx < lim && ny < lim && nz < lim) {
                    const int gn = cid_leaf[morton3(nx, ny, nz)];
                    if (gn >= 0) {
                        st = cstart[gn];
                        ct = ccount[gn];
                    }
                }
                nb_start[lane] = st;
            }
            int x = ct;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane < 27) nb_pre[lane + 1] = x;
            if (lane == 0) nb_pre[0] = 0;
        }
        __syncthreads();
        const int ns = nb_pre[27];
        for (int t0 = tb; t0 < te; t0 += kNfThreads) {   // targets in blocks of 128
            const int ntb = min(kNfThreads, te - t0);
            const int nch = kNfThreads / ntb;            // source chunks per target
            const int ti = tid % ntb, ch = tid / ntb;
            const bool active = ch < nch;
            const R me = sorted[ts + t0 + ti];
            double ex = 0, ey = 0, ez = 0, ph = 0, cex = 0, cey = 0, cez = 0, cph = 0;
            bool first = true;
            for (int s0 = 0; s0 < ns; s0 += kNfSrc64) {    // sources in passes
                const int nsb = min(kNfSrc64, ns - s0);
                __syncthreads();
                for (int j = tid; j < nsb; j += kNfThreads) {
                    const int v = s0 + j;
                    int k = 0;  // largest k with nb_pre[k] <= v (binary search over 28 bounds)
#pragma unroll
                    for (int step = 16; step > 0; step >>= 1)
                        if (k + step <= 26 && nb_pre[k + step] <= v) k += step;
                    const int dx = k / 9 - 1, dy = (k / 3) % 3 - 1, dz = k % 3 - 1;
                    src[j] = Ion<double>::shifted(sorted[nb_start[k] + (v - nb_pre[k])], dx, dy, dz);
                }
                __syncthreads();
                if (active) {
                    // the target's own entry: leaf offset d = 0 is neighbour 13
                    const int self = nb_pre[13] + (t0 + ti) - s0;
                    for (int jb = ch; jb < nsb; jb += 64 * nch) {
                        const int je = min(nsb, jb + 64 * nch);
                        double px = 0, py = 0, pz = 0, pp = 0;
#pragma unroll 2
                        for (int j = jb; j < je; j += nch) {
                            if (j == self) continue;
                            double rx, ry, rz, q;
                            Ion<double>::sep_shifted(me, src[j], rx, ry, rz, q);
                            const double ir = rsqrt(rx * rx + ry * ry + rz * rz);
                            const double qi = q * ir;
                            const double q3 = qi * (ir * ir);
                            px += q3 * rx;
                            py += q3 * ry;
                            pz += q3 * rz;
                            if (PHI) pp += qi;
                        }
                        if (first) {  // the compensated sum of one term is that term
                            ex = px;
                            ey = py;
                            ez = pz;
                            ph = pp;
                            first = false;
                        } else {
                            kb_add(ex, cex, px);
                            kb_add(ey, cey, py);
                            kb_add(ez, cez, pz);
                            if (PHI) kb_add(ph, cph, pp);
                        }
                    }
                }
            }
            if (ns > 64 * nch || ns > kNfSrc64) {  // more than one block of sources somewhere
                ex += cex;
                ey += cey;
                ez += cez;
                ph += cph;
            }
            __syncthreads();  // the sources are read
            part[tid] = make_double4_32a(ex, ey, ez, ph);
            __syncthreads();
            // the chunks in order, compensated: a thread per target and component
            const double* p = reinterpret_cast<const double*>(part);
            for (int e = tid; e < 4 * ntb; e += kNfThreads) {
                double s = 0, c = 0;
                for (int k = 0; k < nch; ++k) kb_add_d(s, c, p[4 * ntb * k + e]);
                near[4 * (int64_t)(ts + t0) + e] = s + c;
            }
            __syncthreads();
        }
    }
}

// L2P (Eq. L2P) and the total field, one block per target leaf.
//   * Per leaf, four derived expansions are formed in shared memory from the
//     leaf's local expansion L: for every (n, m) a pair D_k(n, m) such that
//     the potential and the three gradient components are sums over (n, m)
//     of Re D_k Y^_n^m + Im D_k Im Y^_n^m -- the terms of l2p_eval_cols regrouped
//     by the harmonic they multiply (D_phi = w L_{n,m}; D_z = w e L_{n+1,m};
//     D_x, D_y from f L_{n+1,m+1} and g L_{n+1,m-1}).  The leaf's ~10 targets
//     share them.
//   * One target per 16-lane half-warp, lane m holding column m: the
//     diagonal Y^_m^m = prod_{k<=m} (x + i y) c_k is an inclusive prefix
//     product over the lanes (4 shuffle steps), then lane m runs its column
//     recurrence n = m..p adding four dot products per step; a fixed shuffle
//     tree sums the columns (deterministic).
// The near field (if any) is added and the field written in the original ion
// order scaled to SI (k_e / s^2 for E, k_e / s for phi, s = leaf side).
constexpr int kL2pThreads = 128;


// The derived expansions of one local expansion Lr (see k_l2p) at (nn, mm):
// put(k, phi, grad x, grad y, grad z) for the real part and, for mm > 0, the
// imaginary part (for mm = 0 it would meet Im Y = 0).
template <typename T, class Put>
__device__ __forceinline__ void l2p_derive_entry(int p, int nn, int mm, const T* Lr,
                                                 const HarmTables<T>& t, Put put) {
    const int k = re_idx(nn, mm);
    const T w = mm > 0 ? T(2) : T(1);
    T d0r = w * Lr[k], d0i = mm > 0 ? w * Lr[k + 1] : T(0);
    T dxr = 0, dxi = 0, dyr = 0, dyi = 0, dzr = 0, dzi = 0;
    if (nn + 1 <= p) {
        const int k1 = re_idx(nn + 1, mm);
        const T e = w * t.e[nn][mm];
        dzr = e * Lr[k1];
        dzi = mm > 0 ? e * Lr[k1 + 1] : T(0);
        const int k2 = re_idx(nn + 1, mm + 1);
        const T f = t.f[nn][mm], l2r = Lr[k2], l2i = Lr[k2 + 1];
        dxr = f * l2r;
        dxi = f * l2i;
        dyr = f * l2i;
        dyi = -f * l2r;
        if (mm >= 1) {
            const int k3 = re_idx(nn + 1, mm - 1);
            const T gg = t.g[nn][mm], l3r = Lr[k3], l3i = mm - 1 > 0 ? Lr[k3 + 1] : T(0);
            dxr -= gg * l3r;
            dxi -= gg * l3i;
            dyr += gg * l3i;
            dyi -= gg * l3r;
        }
    }
    put(k, d0r, dxr, dyr, dzr);
    if (mm > 0) put(k + 1, d0i, dxi, dyi, dzi);
}
// all of them into D4[4][P], by the block's threads
template <typename T>
__device__ __forceinline__ void l2p_derive(int p, const T* Lr, const HarmTables<T>& t, T (*D4)[kPmax]) {
    const int C = p + 1;
    for (int q = threadIdx.x; q < C * C; q += kL2pThreads) {
        const int nn = q / C, mm = q % C;
        if (mm > nn) continue;
        l2p_derive_entry<T>(p, nn, mm, Lr, t, [&](int k, T a, T b, T c, T d) {
            D4[0][k] = a;
            D4[1][k] = b;
            D4[2][k] = c;
            D4[3][k] = d;
        });
    }
}

// column m of the potential and gradient at (x, y, z) from derived
// expansions D4; every lane of the half-warp calls it (the prefix product
// shuffles), lanes m > p return zeros.  At p = 16 the last column (m = 16,
// degree 16 only) goes to lane 15 beside its own.
template <typename T>
__device__ __forceinline__ void l2p_columns(int p, int m, unsigned hw_mask, T x, T y, T z,
                                            const HarmTables<T>& t, const T (*D4)[kPmax], T& ph,
                                            T& ax, T& ay, T& az) {
    // diagonal: inclusive prefix product of (x + i y) c_k over k = 1..m
    T dre = m == 0 ? T(1) : x * t.c[m <= p ? m : 0];
    T dim = m == 0 ? T(0) : y * t.c[m <= p ? m : 0];
#pragma unroll
    for (int off = 1; off < 16; off <<= 1) {
        const T ore = __shfl_up_sync(hw_mask, dre, off, 16);
        const T oim = __shfl_up_sync(hw_mask, dim, off, 16);
        if (m >= off) {
            const T r = ore * dre - oim * dim;
            dim = ore * dim + oim * dre;
            dre = r;
        }
    }
    ph = ax = ay = az = T(0);
    if (m > p) return;
    const T r2 = x * x + y * y + z * z;
    T yr = dre, yi = dim, y1r = 0, y1i = 0;  // Y_n^m, Y_{n-1}^m
    for (int nn = m; nn <= p; ++nn) {
        if (nn == m + 1) {
            y1r = yr;
            y1i = yi;
            yr = z * t.d[m] * y1r;
            yi = z * t.d[m] * y1i;
        } else if (nn > m + 1) {
            const T a = t.a[nn][m] * z, b = t.b[nn][m] * r2;
            const T cr = a * yr - b * y1r, ci = a * yi - b * y1i;
            y1r = yr;
            y1i = yi;
            yr = cr;
            yi = ci;
        }
        const int k = re_idx(nn, m);
        ph += D4[0][k] * yr;
        ax += D4[1][k] * yr;
        ay += D4[2][k] * yr;
        az += D4[3][k] * yr;
        if (m > 0) {
            ph += D4[0][k + 1] * yi;
            ax += D4[1][k + 1] * yi;
            ay += D4[2][k + 1] * yi;
            az += D4[3][k + 1] * yi;
        }
    }
    if (p == 16 && m == 15) {
        // Y_16^16 = c_16 (x + i y) Y_15^15, the one term of column 16
        const T gr = (dre * x - dim * y) * t.c[16], gi = (dre * y + dim * x) * t.c[16];
        const int k = re_idx(16, 16);
        ph += D4[0][k] * gr + D4[0][k + 1] * gi;
        ax += D4[1][k] * gr + D4[1][k + 1] * gi;
        ay += D4[2][k] * gr + D4[2][k + 1] * gi;
        az += D4[3][k] * gr + D4[3][k + 1] * gi;
    }
}

// The same sums on an 8-lane group (p <= 15): lane j takes column j and, if
// p - j > j, column p - j, about p + 2 recurrence steps on every lane instead
// of p + 1 - m on a lane per column (on 16 lanes half the lane steps idle).
// Diagonals: lanes hold w_j = (x + i y) c_j and w_{8+j}; two inclusive prefix
// products over the group give Y_j^j and prod_{k=8..8+j} w_k, and Y_m^m for
// m >= 8 is Y_7^7 times the latter (one more rounding than the sequential
// product; every lane fetches its second diagonal by one shuffle).
template <typename T>
__device__ __forceinline__ void l2p_col_run(int p, int m, T yr, T yi, T z, T r2,
                                            const HarmTables<T>& t, const T (*D4)[kPmax], T& ph,
                                            T& ax, T& ay, T& az) {
    T y1r = 0, y1i = 0;  // Y_{n-1}^m
    for (int nn = m; nn <= p; ++nn) {
        if (nn == m + 1) {
            y1r = yr;
            y1i = yi;
            yr = z * t.d[m] * y1r;
            yi = z * t.d[m] * y1i;
        } else if (nn > m + 1) {
            const T a = t.a[nn][m] * z, b = t.b[nn][m] * r2;
            const T cr = a * yr - b * y1r, ci = a * yi - b * y1i;
            y1r = yr;
            y1i = yi;
            yr = cr;
            yi = ci;
        }
        const int k = re_idx(nn, m);
        ph += D4[0][k] * yr;
        ax += D4[1][k] * yr;
        ay += D4[2][k] * yr;
        az += D4[3][k] * yr;
        if (m > 0) {
            ph += D4[0][k + 1] * yi;
            ax += D4[1][k + 1] * yi;
            ay += D4[2][k + 1] * yi;
            az += D4[3][k + 1] * yi;
        }
    }
}

template <typename T>
__device__ __forceinline__ void l2p_columns8(int p, int j, unsigned gmask, T x, T y, T z,
                                             const HarmTables<T>& t, const T (*D4)[kPmax], T& ph,
                                             T& ax, T& ay, T& az) {
    T ar = T(1), ai = T(0), br = T(1), bi = T(0);
    if (j >= 1 && j <= p) {
        ar = x * t.c[j];
        ai = y * t.c[j];
    }
    if (8 + j <= p) {
        br = x * t.c[8 + j];
        bi = y * t.c[8 + j];
    }
#pragma unroll
    for (int off = 1; off < 8; off <<= 1) {
        const T oar = __shfl_up_sync(gmask, ar, off, 8), oai = __shfl_up_sync(gmask, ai, off, 8);
        const T obr = __shfl_up_sync(gmask, br, off, 8), obi = __shfl_up_sync(gmask, bi, off, 8);
        if (j >= off) {
            const T r = oar * ar - oai * ai;
            ai = oar * ai + oai * ar;
            ar = r;
            const T s2 = obr * br - obi * bi;
            bi = obr * bi + obi * br;
            br = s2;
        }
    }
    const T d7r = __shfl_sync(gmask, ar, 7, 8), d7i = __shfl_sync(gmask, ai, 7, 8);
    const T er = d7r * br - d7i * bi, ei = d7r * bi + d7i * br;  // Y_{8+j}^{8+j}
    const int m2 = p - j;
    const int src = m2 >= 8 ? m2 - 8 : (m2 >= 0 ? m2 : 0);
    const T gar = __shfl_sync(gmask, ar, src, 8), gai = __shfl_sync(gmask, ai, src, 8);
    const T ger = __shfl_sync(gmask, er, src, 8), gei = __shfl_sync(gmask, ei, src, 8);
    ph = ax = ay = az = T(0);
    const T r2 = x * x + y * y + z * z;
    if (j <= m2) l2p_col_run<T>(p, j, ar, ai, z, r2, t, D4, ph, ax, ay, az);
    if (m2 > j)
        l2p_col_run<T>(p, m2, m2 >= 8 ? ger : gar, m2 >= 8 ? gei : gai, z, r2, t, D4, ph, ax, ay,
                       az);
}

// nlev = 2: the leaf's expansion holds its own M2L sum only, and the
// parent's complete expansion is evaluated at the ion in the parent's frame
// (equal to the L2L shift into the leaf, which shifts a truncated expansion
// exactly), saving the last L2L launch.
template <typename T, int G>
__device__ __forceinline__ void k_l2p_body(
    const BlockId& blk, int64_t n, int D, int p, int ld, bool far, int nlev, const RootCube* root,
    const LevelInfo* linfo, const uint32_t* __restrict__ code, const int32_t* __restrict__ cid,
    const typename Ion<T>::rec* __restrict__ sorted, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ cstart, const int32_t* __restrict__ ccount,
    const T* __restrict__ L, const T* __restrict__ near, double* E, double* phi) {
    pdl_wait();
    const int g0 = linfo->gbase[D], g1 = linfo->gbase[D + 1];
    if (g0 + (int)blk.x >= g1) return;  // no leaf for this block
    constexpr int NL = sizeof(T) == 4 ? 3 : 2;  // levels evaluated at most (shared memory)
    __shared__ T sL[NL][kPmax];
    __shared__ T sD[NL][4][kPmax];  // derived expansions: phi, grad x, grad y, grad z
    __shared__ HarmTables<T> t;
    __shared__ double s_f[2];
    {
        const int* src = reinterpret_cast<const int*>(&gtab<T>());
        int* dst = reinterpret_cast<int*>(&t);
        for (int i = threadIdx.x; i < (int)(sizeof(HarmTables<T>) / sizeof(int)); i += kL2pThreads)
            dst[i] = src[i];
    }
    // SI scale factors, once per block: FP64 division is slow on this GPU,
    // and every thread computing them cost more than the L2P itself
    if (threadIdx.x == 0) {
        const double sl = root->side / (double)(1 << D);
        s_f[0] = kCoulomb / (sl * sl);
        s_f[1] = kCoulomb / sl;
    }
    __syncthreads();
    const T tE = (T)s_f[0], tP = (T)s_f[1];
    // a group of G lanes per target: G = 8 (p <= 15, l2p_columns8) or 16
    const int lane = threadIdx.x & 31, m = lane & (G - 1);
    const int slot_in_pass = threadIdx.x / G;         // target of this group
    constexpr int kPerPass = kL2pThreads / G;
    const unsigned hw_mask = (G == 8 ? 0xffu : 0xffffu) << (lane & (32 - G));
    const int P = (p + 1) * (p + 1);
    const int levs = far ? (nlev < NL ? nlev : NL) : 0;
    for (int g = g0 + (int)blk.x; g < g1; g += (int)blk.nx) {
        const int ts = cstart[g], nt = ccount[g];
        const uint32_t cl = code[g];
        int ix, iy, iz;
        demorton3(cl, ix, iy, iz);
        __syncthreads();  // sL, sD free from the previous leaf
        for (int lv = 0; lv < levs; ++lv) {
            // dense maps of levels 2.. concatenated: level l starts at (8^l - 64) / 7
            const int ga =
                lv == 0 ? g : cid[(((1ll << (3 * (D - lv))) - 64) / 7) + (cl >> (3 * lv))];
            for (int c = threadIdx.x; c < P; c += kL2pThreads) sL[lv][c] = L[(int64_t)ga * ld + c];
        }
        __syncthreads();
        for (int lv = 0; lv < levs; ++lv) l2p_derive<T>(p, sL[lv], t, sD[lv]);
        __syncthreads();
        for (int t0 = 0; t0 < nt; t0 += kPerPass) {
            const int ti = t0 + slot_in_pass;
            if (ti >= nt) continue;  // whole groups only: the shuffles stay within one
            T ex = 0, ey = 0, ez = 0, ph = 0;
            const typename Ion<T>::rec me = sorted[ts + ti];
            for (int lv = 0; lv < levs; ++lv) {
                T x, y, z, q;
                const int am = (1 << lv) - 1;  // the leaf's position inside the ancestor
                ion_in_ancestor(me, lv, ix & am, iy & am, iz & am, x, y, z, q);
                T cph, cax, cay, caz;
                if (G == 8) l2p_columns8<T>(p, m, hw_mask, x, y, z, t, sD[lv], cph, cax, cay, caz);
                else l2p_columns<T>(p, m, hw_mask, x, y, z, t, sD[lv], cph, cax, cay, caz);
                // level units -> leaf units: phi / 2^lv, E / 4^lv (exact)
                const T fp1 = lv == 0 ? T(1) : (lv == 1 ? T(0.5) : T(0.25)), fe1 = fp1 * fp1;
                ph += fp1 * cph;
                ex -= fe1 * cax;
                ey -= fe1 * cay;
                ez -= fe1 * caz;
            }
            // column sums: a fixed shuffle tree over the group
#pragma unroll
            for (int off = G / 2; off > 0; off >>= 1) {
                ex += __shfl_xor_sync(hw_mask, ex, off, G);
                ey += __shfl_xor_sync(hw_mask, ey, off, G);
                ez += __shfl_xor_sync(hw_mask, ez, off, G);
                ph += __shfl_xor_sync(hw_mask, ph, off, G);
            }
            if (m == 0) {
                // near + far and the SI scale in T: in FP32 one conversion per
                // stored component (FP64 instructions are scarce on this GPU)
                if (near) {
                    const T* o = near + 4 * (int64_t)(ts + ti);
                    ex += o[0];
                    ey += o[1];
                    ez += o[2];
                    ph += o[3];
                }
                const int i = perm[ts + ti];
                E[i] = (double)(tE * ex);
                E[n + i] = (double)(tE * ey);
                E[2 * n + i] = (double)(tE * ez);
                if (phi) phi[i] = (double)(tP * ph);
            }
        }
    }
}
template <typename T, int G>
__global__ void __launch_bounds__(kL2pThreads) k_l2p(
    int64_t n, int D, int p, int ld, bool far, int nlev, const RootCube* root,
    const LevelInfo* linfo, const uint32_t* __restrict__ code, const int32_t* __restrict__ cid,
    const typename Ion<T>::rec* __restrict__ sorted, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ cstart, const int32_t* __restrict__ ccount,
    const T* __restrict__ L, const T* __restrict__ near, double* E, double* phi) {
    k_l2p_body<T, G>(solo_block(), n, D, p, ld, far, nlev, root, linfo, code, cid, sorted, perm, cstart,
                     ccount, L, near, E, phi);
}

// L2P in FP64 (see k_p2m_f64): a thread per ion, the derived expansions of
// up to `lmax` leaves in shared memory (leaf strides odd in 8-byte units: the
// leaves of a warp read different banks).  PHI: the potential too.
constexpr int kL2pLeaves = 16;
// leaves whose expansions (derived 4 x, local 1 x) fit about 100 KB
inline int l2p_f64_leaves(int P) {
    const int l = 100 * 1024 / (5 * P * 8 + 8);
    return l < 4 ? 4 : (l > kL2pLeaves ? kL2pLeaves : l);
}
inline size_t l2p_f64_smem(int P) { return sizeof(double) * (size_t)l2p_f64_leaves(P) * (5 * P + 1); }

template <bool PHI>
__global__ void __launch_bounds__(kSlotThreads) k_l2p_f64(
    int64_t n, int D, int p, int ld, int lmax, const RootCube* root,
    const int32_t* __restrict__ leaf_of, const int32_t* __restrict__ cstart,
    const int32_t* __restrict__ ccount, const Ion<double>::rec* __restrict__ sorted,
    const int32_t* __restrict__ perm, const double* __restrict__ L,
    const double* __restrict__ near, double* E, double* phi) {
    extern __shared__ double slot_smem[];  // derived [lmax][4 P + 1], local [lmax][P]
    __shared__ int s_g[kL2pLeaves], s_cnt[2], s_new[2];
    __shared__ uint16_t s_nm[(kMaxOrder + 1) * (kMaxOrder + 2) / 2];
    __shared__ double s_f[2];
    const int P = (p + 1) * (p + 1), DS = 4 * P + 1, tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    double* sD = slot_smem;
    double* sL = slot_smem + lmax * DS;
    const int NT = (p + 1) * (p + 2) / 2;
    for (int nn = tid; nn <= p; nn += kSlotThreads)
        for (int m = 0; m <= nn; ++m) s_nm[nn * (nn + 1) / 2 + m] = (uint16_t)(nn << 8 | m);
    pdl_wait();
    int s0, s1;
    if (!slot_window(n, blockIdx.x, leaf_of, cstart, ccount, s0, s1)) return;  // uniform
    if (tid == 0) {
        const double inv = 1.0 / (root->side / (double)(1 << D));
        s_f[0] = kCoulomb * (inv * inv);
        s_f[1] = kCoulomb * inv;
    }
    for (int p0 = s0; p0 < s1;) {
        // the pass: slots p0 .. p0 + ni - 1, at most 64 and of at most lmax leaves
        const bool live = p0 + tid < s1;
        const int g = live ? leaf_of[p0 + tid] : -1;
        const bool head = live && (tid == 0 || leaf_of[p0 + tid - 1] != g);
        const unsigned bal = __ballot_sync(0xffffffffu, head);
        __syncthreads();  // the previous pass is done with the shared arrays
        if (lane == 0) s_new[wid] = __popc(bal);
        __syncthreads();
        const int ord = (wid ? s_new[0] : 0) + __popc(bal & (0xffffffffu >> (31 - lane))) - 1;
        const bool in = live && ord < lmax;
        if (head && in) s_g[ord] = g;
        const unsigned inb = __ballot_sync(0xffffffffu, in);
        if (lane == 0) s_cnt[wid] = __popc(inb);
        __syncthreads();
        const int ni = s_cnt[0] + s_cnt[1], nl = min(lmax, s_new[0] + s_new[1]);
        for (int l = 0; l < nl; ++l)
            for (int c = tid; c < P; c += kSlotThreads) sL[l * P + c] = L[(int64_t)s_g[l] * ld + c];
        __syncthreads();
        for (int u = tid; u < nl * NT; u += kSlotThreads) {
            const int l = u / NT, nm = s_nm[u - l * NT];
            double* d = sD + l * DS;
            l2p_derive_entry<double>(p, nm >> 8, nm & 255, sL + l * P, g_tab_d,
                                     [&](int k, double a, double b, double c, double e) {
                                         d[k] = a;
                                         d[P + k] = b;
                                         d[2 * P + k] = c;
                                         d[3 * P + k] = e;
                                     });
        }
        __syncthreads();
        if (in) {
            const double* D4 = sD + ord * DS;
            double x, y, z, q, ph = 0, ax = 0, ay = 0, az = 0;
            Ion<double>::get(sorted[p0 + tid], x, y, z, q);
            for_each_ups<double>(p, x, y, z, c_tab_d, [&](int nn, int m, double yr, double yi) {
                const double* d = D4 + re_idx(nn, m);
                if (PHI) ph += d[0] * yr;
                ax += d[P] * yr;
                ay += d[2 * P] * yr;
                az += d[3 * P] * yr;
                if (m > 0) {
                    if (PHI) ph += d[1] * yi;
                    ax += d[P + 1] * yi;
                    ay += d[2 * P + 1] * yi;
                    az += d[3 * P + 1] * yi;
                }
            });
            double ex = -ax, ey = -ay, ez = -az;
            if (near) {
                const Ion<double>::rec o = *reinterpret_cast<const Ion<double>::rec*>(near + 4 * (int64_t)(p0 + tid));
                ex += o.x;
                ey += o.y;
                ez += o.z;
                if (PHI) ph += o.w;
            }
            const int i = perm[p0 + tid];
            E[i] = s_f[0] * ex;
            E[n + i] = s_f[0] * ey;
            E[2 * n + i] = s_f[0] * ez;
            if (PHI) phi[i] = s_f[1] * ph;
        }
        p0 += ni;
    }
}

// L2P in FP32 (p <= 15): G = 1 or 4 threads per ion, a block for the ions of a
// window of sorted slots as in k_l2p_f64; the leaf's, its parent's and
// grandparent's derived expansions (nlev of them) once per block for all the
// leaves that share them, as one float4 (phi, grad) per coefficient.  With 8
// lanes to an ion and a block per leaf (k_l2p) a recurrence step served four
// ions, each leaf derived its ancestors' expansions anew and leaves of few
// ions left most of a block idle.  Every sum is formed as there: the diagonals
// by the same tree of products, "lane" g = 0 .. 7 of an ion adds columns g and
// p - g of every level in turn, and the eight sums join pairwise (0 + 4,
// 2 + 6, ...), so the fields are the same bit for bit.
//
// Bound by the latency of the chains of fused multiply-adds and shared loads
// at few warps per SM: two columns run side by side (1,500 -> 820 us at 1e6
// ions, p = 12, with blocks of 64 threads and 36 KB), and a block of 128 ions
// shares more ancestors than two of 64 (820 -> 700 us; 72 KB a block, as at 36
// KB many blocks need a second pass).  In all 1,727 -> 700 us at 1e6 ions,
// 220 -> 115 us at 1e5 (p = 12), 42 -> 22 us at 23,000 (p = 8).
// Small crystals lack the ions to fill the chip with one thread each: four,
// each with two of the eight sums, and blocks of 64 ions for windows of 28, so
// that nearly all need a single pass (10,000 ions, p = 12: 31 -> 21 us; with
// blocks of 32 ions 27, with windows of 16 33).
constexpr int kL2pExp = 64;  // expansions per pass at most
__host__ __device__ inline constexpr int l2p_f32_threads(int G) { return G == 1 ? 128 : 256; }
__host__ __device__ inline constexpr int l2p_f32_window(int G) { return G == 1 ? 112 : 28; }
// expansions (derived 16 bytes a coefficient, local 4) that fit 72 or 56 KB
inline int l2p_f32_exps(int P, int G) {
    const int l = (G == 1 ? 72 : 56) * 1024 / (20 * P);
    return l < 8 ? 8 : (l > kL2pExp ? kL2pExp : l);
}
inline size_t l2p_f32_smem(int P, int G) { return (size_t)l2p_f32_exps(P, G) * P * 20 + 16; }

struct L2pSum {
    float ph, ax, ay, az;
};
// one column's running harmonic: Y_nn^m and Y_{nn-1}^m
struct L2pCol {
    float yr, yi, y1r, y1i;
    __device__ __forceinline__ void second(int m, float z) {
        y1r = yr;
        y1i = yi;
        yr = z * c_tab_f.d[m] * y1r;
        yi = z * c_tab_f.d[m] * y1i;
    }
    __device__ __forceinline__ void next(int nn, int m, float z, float r2) {
        const float a = c_tab_f.a[nn][m] * z, b = c_tab_f.b[nn][m] * r2;
        const float cr = a * yr - b * y1r, ci = a * yi - b * y1i;
        y1r = yr;
        y1i = yi;
        yr = cr;
        yi = ci;
    }
    __device__ __forceinline__ void add(int nn, int m, const float4* D4, L2pSum& s) const {
        const int k = re_idx(nn, m);
        const float4 dr = D4[k];
        s.ph += dr.x * yr;
        s.ax += dr.y * yr;
        s.ay += dr.z * yr;
        s.az += dr.w * yr;
        if (m > 0) {
            const float4 di = D4[k + 1];
            s.ph += di.x * yi;
            s.ax += di.y * yi;
            s.ay += di.z * yi;
            s.az += di.w * yi;
        }
    }
};
__device__ __forceinline__ void l2p_run(int p, int m, float2 diag, float z, float r2,
                                        const float4* D4, L2pSum& s) {
    L2pCol c{diag.x, diag.y, 0.f, 0.f};
    c.add(m, m, D4, s);
    if (m == p) return;
    c.second(m, z);
    c.add(m + 1, m, D4, s);
    for (int nn = m + 2; nn <= p; ++nn) {
        c.next(nn, m, z, r2);
        c.add(nn, m, D4, s);
    }
}
// columns m (into a) and m + 1 <= p (into b) side by side: two chains in flight
__device__ __forceinline__ void l2p_run2(int p, int m, float2 da, float2 db, float z, float r2,
                                         const float4* D4, L2pSum& a, L2pSum& b) {
    L2pCol u{da.x, da.y, 0.f, 0.f}, v{db.x, db.y, 0.f, 0.f};
    u.add(m, m, D4, a);
    u.second(m, z);
    u.add(m + 1, m, D4, a);
    v.add(m + 1, m + 1, D4, b);
    if (m + 2 > p) return;
    u.next(m + 2, m, z, r2);
    v.second(m + 1, z);
    u.add(m + 2, m, D4, a);
    v.add(m + 2, m + 1, D4, b);
    for (int nn = m + 3; nn <= p; ++nn) {
        u.next(nn, m, z, r2);
        v.next(nn, m + 1, z, r2);
        u.add(nn, m, D4, a);
        v.add(nn, m + 1, D4, b);
    }
}

template <int G>
__device__ __forceinline__ void k_l2p_f32_body(
    const BlockId& blk, int64_t n, int D, int p, int ld, int nlev, int emax, const RootCube* root,
    const uint32_t* __restrict__ code, const int32_t* __restrict__ cid,
    const int32_t* __restrict__ leaf_of, const int32_t* __restrict__ cstart,
    const int32_t* __restrict__ ccount, const Ion<float>::rec* __restrict__ sorted,
    const int32_t* __restrict__ perm, const float* __restrict__ L,
    const float* __restrict__ near, double* E, double* phi) {
    extern __shared__ float4 l2p_smem[];  // derived [emax][P], then local [emax][P] floats
    __shared__ int s_row[kL2pExp], s_new[3][l2p_f32_threads(G) / 32], s_cnt[l2p_f32_threads(G) / 32], s_tot[3];
    __shared__ uint16_t s_nm[(kMaxOrder + 1) * (kMaxOrder + 2) / 2];
    __shared__ double s_f[2];
    const int P = (p + 1) * (p + 1), tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
    const int u0 = tid / G, part = tid % G;  // the thread's ion of the pass, and its share
    const int NT = (p + 1) * (p + 2) / 2;
    float4* sD = l2p_smem;
    float* sL = reinterpret_cast<float*>(l2p_smem + emax * P);
    for (int nn = tid; nn <= p; nn += l2p_f32_threads(G))
        for (int m = 0; m <= nn; ++m) s_nm[nn * (nn + 1) / 2 + m] = (uint16_t)(nn << 8 | m);
    pdl_wait();
    int s0, s1;
    if (!slot_window(n, (int)blk.x, leaf_of, cstart, ccount, s0, s1, l2p_f32_window(G))) return;  // uniform
    if (tid == 0) {
        const double sl = root->side / (double)(1 << D);
        s_f[0] = kCoulomb / (sl * sl);
        s_f[1] = kCoulomb / sl;
    }
    for (int p0 = s0; p0 < s1;) {
        // the pass: at most l2p_f32_threads(G) / G slots whose cells number at most emax
        const bool live = p0 + u0 < s1;
        const int g = live ? leaf_of[p0 + u0] : -1;
        const uint32_t cl = live ? code[g] : 0xffffffffu;
        const uint32_t prev = u0 == 0 || !live ? 0xffffffffu : code[leaf_of[p0 + u0 - 1]];
        unsigned bal[3];
        bool head[3];
#pragma unroll
        for (int lv = 0; lv < 3; ++lv) {
            head[lv] = live && part == 0 && lv < nlev && (u0 == 0 || (prev >> (3 * lv)) != (cl >> (3 * lv)));
            bal[lv] = __ballot_sync(0xffffffffu, head[lv]);
        }
        __syncthreads();  // the previous pass is done with the shared arrays
        if (lane == 0)
            for (int lv = 0; lv < 3; ++lv) s_new[lv][wid] = __popc(bal[lv]);
        if (tid < 3) s_tot[tid] = 0;
        __syncthreads();
        int ord[3], used = 0;
#pragma unroll
        for (int lv = 0; lv < 3; ++lv) {
            ord[lv] = __popc(bal[lv] & (0xffffffffu >> (31 - lane))) - 1;
#pragma unroll
            for (int w = 0; w < l2p_f32_threads(G) / 32 - 1; ++w) ord[lv] += w < wid ? s_new[lv][w] : 0;
            used += ord[lv] + 1;
        }
        const bool in = live && used <= emax;
        const unsigned inb = __ballot_sync(0xffffffffu, in && part == 0);
        if (lane == 0) s_cnt[wid] = __popc(inb);
        __syncthreads();
        int ni = 0;
#pragma unroll
        for (int w = 0; w < l2p_f32_threads(G) / 32; ++w) ni += s_cnt[w];
        if (tid == (ni - 1) * G)
            for (int lv = 0; lv < 3; ++lv) s_tot[lv] = ord[lv] + 1;
        __syncthreads();
        int base[3] = {0, s_tot[0], s_tot[0] + s_tot[1]};
        const int ne = base[2] + s_tot[2];
#pragma unroll
        for (int lv = 0; lv < 3; ++lv)
            if (in && head[lv])
                // dense maps of levels 2.. concatenated: level l starts at (8^l - 64) / 7
                s_row[base[lv] + ord[lv]] =
                    lv == 0 ? g : cid[(((1ll << (3 * (D - lv))) - 64) / 7) + (cl >> (3 * lv))];
        __syncthreads();
        for (int e = 0; e < ne; ++e)
            for (int c = tid; c < P; c += l2p_f32_threads(G)) sL[e * P + c] = L[(int64_t)s_row[e] * ld + c];
        __syncthreads();
        for (int u = tid; u < ne * NT; u += l2p_f32_threads(G)) {
            const int e = u / NT, nm = s_nm[u - e * NT];
            float4* d = sD + e * P;
            l2p_derive_entry<float>(p, nm >> 8, nm & 255, sL + e * P, g_tab_f,
                                    [&](int k, float a, float b, float c, float w) {
                                        d[k] = make_float4(a, b, c, w);
                                    });
        }
        __syncthreads();
        if (in) {
            const Ion<float>::rec me = sorted[p0 + u0];
            int ix, iy, iz;
            demorton3(cl, ix, iy, iz);
            constexpr int NV = 8 / G;  // of the eight partial sums: part NV .. part NV + NV - 1
            float vx[NV], vy[NV], vz[NV], vp[NV];
#pragma unroll
            for (int q = 0; q < NV; ++q) vx[q] = vy[q] = vz[q] = vp[q] = 0.f;
#pragma unroll 1
            for (int lv = 0; lv < nlev; ++lv) {
                const float4* D4 = sD + (base[lv] + ord[lv]) * P;
                float x, y, z, qq;
                const int am = (1 << lv) - 1;  // the leaf's position inside the ancestor
                ion_in_ancestor(me, lv, ix & am, iy & am, iz & am, x, y, z, qq);
                // diagonals Y_m^m, m = 0 .. 15: two prefix products of eight
                float ar[8], ai[8], br[8], bi[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    ar[q] = br[q] = 1.f;
                    ai[q] = bi[q] = 0.f;
                    if (q >= 1 && q <= p) {
                        ar[q] = x * c_tab_f.c[q];
                        ai[q] = y * c_tab_f.c[q];
                    }
                    if (8 + q <= p) {
                        br[q] = x * c_tab_f.c[8 + q];
                        bi[q] = y * c_tab_f.c[8 + q];
                    }
                }
#pragma unroll
                for (int off = 1; off < 8; off <<= 1)
#pragma unroll
                    for (int q = 7; q >= off; --q) {
                        const float oar = ar[q - off], oai = ai[q - off], obr = br[q - off], obi = bi[q - off];
                        const float r = oar * ar[q] - oai * ai[q];
                        ai[q] = oar * ai[q] + oai * ar[q];
                        ar[q] = r;
                        const float s2 = obr * br[q] - obi * bi[q];
                        bi[q] = obr * bi[q] + obi * br[q];
                        br[q] = s2;
                    }
                float2 dg[16];
#pragma unroll
                for (int q = 0; q < 8; ++q) {
                    dg[q] = make_float2(ar[q], ai[q]);
                    dg[8 + q] = make_float2(ar[7] * br[q] - ai[7] * bi[q], ar[7] * bi[q] + ai[7] * br[q]);
                }
                const float r2 = x * x + y * y + z * z;
                const float fp1 = lv == 0 ? 1.f : (lv == 1 ? 0.5f : 0.25f), fe1 = fp1 * fp1;
#pragma unroll
                for (int r = 0; r < NV; r += 2) {
                    const int q = part * NV + r, m2 = p - q;
                    L2pSum c0{0.f, 0.f, 0.f, 0.f}, c1{0.f, 0.f, 0.f, 0.f};
                    if (m2 - 1 > q + 1) {
                        l2p_run2(p, q, dg[q], dg[q + 1], z, r2, D4, c0, c1);
                        l2p_run2(p, m2 - 1, dg[m2 - 1], dg[m2], z, r2, D4, c1, c0);
                    } else {  // the last columns (p < 15)
                        if (q <= m2) l2p_run(p, q, dg[q], z, r2, D4, c0);
                        if (m2 > q) l2p_run(p, m2, dg[m2], z, r2, D4, c0);
                        if (q + 1 <= m2 - 1) l2p_run(p, q + 1, dg[q + 1], z, r2, D4, c1);
                    }
                    // level units -> leaf units: phi / 2^lv, E / 4^lv (exact)
                    vp[r] += fp1 * c0.ph;
                    vx[r] -= fe1 * c0.ax;
                    vy[r] -= fe1 * c0.ay;
                    vz[r] -= fe1 * c0.az;
                    vp[r + 1] += fp1 * c1.ph;
                    vx[r + 1] -= fe1 * c1.ax;
                    vy[r + 1] -= fe1 * c1.ay;
                    vz[r + 1] -= fe1 * c1.az;
                }
            }
            // every lane of the ion gets the sum
            auto join = [&](float (&v)[NV]) {
                if constexpr (G == 1) {
                    return ((v[0] + v[4]) + (v[2] + v[6])) + ((v[1] + v[5]) + (v[3] + v[7]));
                } else {
                    const unsigned mask = 0xfu << (lane & ~3);
#pragma unroll
                    for (int off = 2; off > 0; off >>= 1)
#pragma unroll
                        for (int q = 0; q < 2; ++q) v[q] += __shfl_xor_sync(mask, v[q], off, 4);
                    return v[0] + v[1];
                }
            };
            float ex = join(vx), ey = join(vy), ez = join(vz), ph = join(vp);
            if (near) {
                const float* o = near + 4 * (int64_t)(p0 + u0);
                ex += o[0];
                ey += o[1];
                ez += o[2];
                ph += o[3];
            }
            const float tE = (float)s_f[0], tP = (float)s_f[1];
            const int i = perm[p0 + u0];
            if constexpr (G == 1) {
                E[i] = (double)(tE * ex);
                E[n + i] = (double)(tE * ey);
                E[2 * n + i] = (double)(tE * ez);
                if (phi) phi[i] = (double)(tP * ph);
            } else {
                const float v = part == 0 ? tE * ex : part == 1 ? tE * ey : part == 2 ? tE * ez : tP * ph;
                double* to = part < 3 ? E + part * n : phi;
                if (to) to[i] = (double)v;
            }
        }
        p0 += ni;
    }
}

template <int G>
__global__ void __launch_bounds__(l2p_f32_threads(G)) k_l2p_f32(
    int64_t n, int D, int p, int ld, int nlev, int emax, const RootCube* root,
    const uint32_t* __restrict__ code, const int32_t* __restrict__ cid,
    const int32_t* __restrict__ leaf_of, const int32_t* __restrict__ cstart,
    const int32_t* __restrict__ ccount, const Ion<float>::rec* __restrict__ sorted,
    const int32_t* __restrict__ perm, const float* __restrict__ L,
    const float* __restrict__ near, double* E, double* phi) {
    k_l2p_f32_body<G>(solo_block(), n, D, p, ld, nlev, emax, root, code, cid, leaf_of, cstart, ccount,
                      sorted, perm, L, near, E, phi);
}

// Direct ancestor local expansions (PT_EXPAND_DIRECT): as k_l2p, but every
// thread evaluates its columns of the M2L-only local expansions of the
// target's cells at levels lmin..D, each at the ion in that cell's frame,
// scaled to leaf units; equal to shifting them down by L2L (which shifts a
// truncated local expansion exactly) and evaluating the leaf's.
template <typename T>
__global__ void __launch_bounds__(kNfThreads) k_l2p_anc(
    int64_t n, int D, int lmin, int p, int ld, const RootCube* root, const LevelInfo* linfo,
    const uint32_t* __restrict__ code, const int32_t* __restrict__ cid,
    const typename Ion<T>::rec* __restrict__ sorted, const int32_t* __restrict__ perm,
    const int32_t* __restrict__ cstart, const int32_t* __restrict__ ccount,
    const T* __restrict__ L, const T* __restrict__ near, double* E, double* phi) {
    __shared__ T part[kNfThreads][4];
    const int tid = threadIdx.x;
    const int lim = 1 << D;
    // SI scale factors, once per block: FP64 division is slow on this GPU,
    // and every thread computing them cost more than the L2P itself
    __shared__ double s_f[2];
    if (threadIdx.x == 0) {
        const double sl = root->side / (double)lim;
        s_f[0] = kCoulomb / (sl * sl);
        s_f[1] = kCoulomb / sl;
    }
    __syncthreads();
    const double fE = s_f[0], fP = s_f[1];
    const int g0 = linfo->gbase[D], g1 = linfo->gbase[D + 1];
    for (int g = g0 + blockIdx.x; g < g1; g += gridDim.x) {
        const int ts = cstart[g], nt = ccount[g];
        const uint32_t cl = code[g];
        int ix, iy, iz;
        demorton3(cl, ix, iy, iz);
        for (int t0 = 0; t0 < nt; t0 += kNfThreads) {
            const int ntb = min(kNfThreads, nt - t0);
            const int nch = kNfThreads / ntb;
            const int ti = tid % ntb, ch = tid / ntb;
            T ex = 0, ey = 0, ez = 0, ph = 0;
            if (ch < nch) {
                const typename Ion<T>::rec me = sorted[ts + t0 + ti];
                for (int l = lmin; l <= D; ++l) {
                    const int sh = D - l, mask = (1 << sh) - 1;
                    // dense maps of levels 2.. concatenated: level l starts at (8^l - 64) / 7
                    const int ga =
                        sh == 0 ? g : cid[(((1ll << (3 * l)) - 64) / 7) + (cl >> (3 * sh))];
                    T fphi, gx, gy, gz, ux, uy, uz, uq;
                    ion_in_ancestor(me, sh, ix & mask, iy & mask, iz & mask, ux, uy, uz, uq);
                    l2p_eval_cols<T>(p, L + (int64_t)ga * ld, ux, uy, uz, tab<T>(), ch, nch, fphi,
                                     gx, gy, gz);
                    // level-l units -> leaf units: phi / 2^sh, E / 4^sh (exact)
                    const T fp1 = (T)1 / (T)(1 << sh), fe1 = fp1 * fp1;
                    ex -= fe1 * gx;
                    ey -= fe1 * gy;
                    ez -= fe1 * gz;
                    ph += fp1 * fphi;
                }
            }
            part[tid][0] = ex;
            part[tid][1] = ey;
            part[tid][2] = ez;
            part[tid][3] = ph;
            __syncthreads();
            if (tid < ntb) {
                T sx = 0, sy = 0, sz = 0, sp = 0, cx = 0, cy = 0, cz = 0, cp = 0;
                for (int c = 0; c < nch; ++c) {
                    const int th = c * ntb + tid;
                    kb_add(sx, cx, part[th][0]);
                    kb_add(sy, cy, part[th][1]);
                    kb_add(sz, cz, part[th][2]);
                    kb_add(sp, cp, part[th][3]);
                }
                double fx = (double)(sx + cx), fy = (double)(sy + cy), fz = (double)(sz + cz),
                       fp = (double)(sp + cp);
                if (near) {
                    const T* o = near + 4 * (int64_t)(ts + t0 + tid);
                    fx += (double)o[0];
                    fy += (double)o[1];
                    fz += (double)o[2];
                    fp += (double)o[3];
                }
                const int i = perm[ts + t0 + tid];
                E[i] = fE * fx;
                E[n + i] = fE * fy;
                E[2 * n + i] = fE * fz;
                if (phi) phi[i] = fP * fp;
            }
            __syncthreads();
        }
    }
}

// the near field of `leaves` leaves at most
template <typename T>
static void launch_p2p(int D, int64_t leaves, int leaf_grid, bool phi, Workspace& ws,
                       const int32_t* cid_leaf, T* near, cudaStream_t s);
template <>
void launch_p2p<float>(int D, int64_t, int leaf_grid, bool, Workspace& ws,
                       const int32_t* cid_leaf, float* near, cudaStream_t s) {
    k_p2p<<<leaf_grid, kNfThreads, 0, s>>>(D, ws.linfo, (const Ion<float>::rec*)ws.sorted, ws.code,
                                             cid_leaf, ws.cstart, ws.ccount, near);
}
template <>
void launch_p2p<double>(int D, int64_t leaves, int, bool phi, Workspace& ws,
                        const int32_t* cid_leaf, double* near, cudaStream_t s) {
    // few leaves: several blocks share a leaf's targets, so that a shallow
    // tree (1,000 ions at depth 2: 63 leaves, 223 us with a block per leaf)
    // fills the GPU.  (One or two blocks per SM, to run beside the
    // translations' CTAs: the FP64 latencies then show, 50 and 42 ms against
    // 35 for the evaluation of 1e6 ions at p = 8.)
    const int64_t want = (int64_t)ws.sms * 4;
    const int parts = (int)(leaves >= want ? 1 : (want + leaves - 1) / leaves);
    const int64_t units = leaves * parts, cap = 152 * 16;
    const int grid = (int)(units < cap ? units : cap);
    auto k = phi ? k_p2p_f64<true> : k_p2p_f64<false>;
    k<<<grid, kNfThreads, 0, s>>>(D, parts, ws.linfo, (const Ion<double>::rec*)ws.sorted, ws.code,
                                  cid_leaf, ws.cstart, ws.ccount, near);
}

template <typename T>
static cudaError_t run_fmm(int64_t n, int D, int phases, Workspace& ws, bool use_tc, double* E,
                           double* phi, cudaStream_t s, cudaEvent_t* ev, bool alone) {
    const int p = ws.p, P = ws.P;
    DenseLayout dl = dense_layout(D);
    T* M = (T*)ws.M;
    T* L = (T*)ws.L;
    T* near = (T*)ws.near;
    const bool far = (phases & PT_PHASE_FAR) && D >= 2;
    const bool nf = (phases & PT_PHASE_NEAR) != 0;
    const int64_t leaves = n < ((int64_t)1 << (3 * D)) ? n : ((int64_t)1 << (3 * D));
    const int leaf_grid = (int)(leaves < 152 * 16 ? (leaves > 0 ? leaves : 1) : 152 * 16);
    // The M2L work list and the near field depend on the tree only: with a
    // side stream they run there, beside the main chain.
    const bool fork = far && nf && ws.side != nullptr;
    cudaStream_t sn = fork ? ws.side : s;
    // ancestor expansions of the tensor-core path directly from the ions
    // instead of the M2M / L2L shifts (an option: a cross-check of the shifts)
    const bool direct = far && use_tc && ws.expand == PT_EXPAND_DIRECT;
    // ancestor levels the leaves' L2P evaluates on the tensor-core paths: the
    // leaf, its parent and grandparent (each shift that L2P replaces is one
    // launch fewer; M2L levels start at 2)
    const int l2p_levels = use_tc ? (D - 1 < 3 ? (D - 1 > 1 ? D - 1 : 1) : 3) : 1;
    cudaError_t e;
    if (fork) {
        if ((e = cudaEventRecord(ws.ev_fork, s)) != cudaSuccess) return e;
        if ((e = cudaStreamWaitEvent(sn, ws.ev_fork, 0)) != cudaSuccess) return e;
    }
    // the M2L work list: the tensor-core schedules, and the pair-packed
    // schedule of the CUDA-core paths
    const bool pairs_simt = far && !use_tc && ws.m2l_pairs;
    // FP64: M2M, M2L and L2L on the tensor cores (m2l_f64.cu), the M2L over
    // the pair work list of all targets or of one batch of them after another
    const bool f64 = far && ws.fp64 && ws.f64_tc;
    const bool f64_batched = f64 && ws.f64_batch > 0;
    if (far && (use_tc || pairs_simt)) {
        if ((e = use_tc ? launch_m2l_tc_worklist(n, D, ws, sn)
                        : launch_m2l_pairs_worklist(n, D, ws, sn)) != cudaSuccess)
            return e;
        if (fork && (e = cudaEventRecord(ws.ev_items, sn)) != cudaSuccess) return e;
    }
    // Multipoles from the ions: at the leaves, and on the tensor-core path also
    // at their parents (a parent holds about eight leaves' ions, cheaper to
    // expand directly than one more M2M launch and its reduction), or at every
    // level >= 2 in the direct mode; M2M shifts the rest up.
    const int lmin_p2m = direct ? 2 : (far && use_tc && D >= 3 ? D - 1 : D);
    // BF16x3: the multipoles' bf16 pieces, the M2L operand, are written by
    // their producers (P2M and the small-level M2M); a split pass covers the
    // levels of the tensor-core M2M (3 .. lmin_p2m - 1)
    uint16_t* Mp = use_tc && ws.tc_bf16 ? ws.M_pieces : nullptr;
    const int split_last = use_tc && ws.tc_bf16 && !direct ? lmin_p2m - 1 : 0;
    if (far && lmin_p2m < D) {
        int64_t cells = 0;
        for (int l = lmin_p2m; l <= D; ++l)
            cells += n < ((int64_t)1 << (3 * l)) ? n : ((int64_t)1 << (3 * l));
        const int grid = (int)(cells < 152 * 16 ? cells : 152 * 16);
        if ((e = launch_pdl(k_p2m_anc<T>, dim3(grid), dim3(kP2mThreads), kP2mAncIons * P * sizeof(T),
                            s, D, lmin_p2m, p, ws.ld, (const LevelInfo*)ws.linfo,
                            (const uint32_t*)ws.code, (const int32_t*)ws.leaf_start,
                            (const int32_t*)ws.leaf_of, (const typename Ion<T>::rec*)ws.sorted,
                            M, Mp)) != cudaSuccess)
            return e;
    } else if (far && sizeof(T) == 8 && n >= kP2mSlotIons) {
        if ((e = launch_pdl(k_p2m_f64, dim3((unsigned)((n + kSlotWindow - 1) / kSlotWindow)),
                            dim3(kSlotThreads), sizeof(double) * kSlotThreads * p2m_f64_stride(P), s, n,
                            p, ws.ld, (const int32_t*)ws.leaf_of, (const int32_t*)ws.cstart,
                            (const int32_t*)ws.ccount, (const Ion<double>::rec*)ws.sorted,
                            (double*)ws.M)) != cudaSuccess)
            return e;
    } else if (far) {
        k_p2m<T><<<leaf_grid, kP2mThreads, kP2mIons * P * sizeof(T), s>>>(
            D, p, ws.ld, ws.linfo, ws.cstart, ws.ccount, (const typename Ion<T>::rec*)ws.sorted, M,
            Mp);
        if ((e = cudaGetLastError()) != cudaSuccess) return e;
    }
    // P2P on the side stream: after P2M on the CUDA-core paths (beside their
    // M2L); on the tensor-core path after the M2L kernel, which needs every
    // SM, beside the slab reduction and the L2L launches, which use few
    // On the tensor-core paths the near field takes a third stream from the
    // fork, beside the upward pass and the work list (both latency-bound).
    // So it does on the FP64 path with the tensor-core translations (10k-ion
    // step 0.77 against 0.71 ms; 1e5-ion evaluation 8.39 against 8.29 ms).
    const bool near_early = fork && (use_tc || f64) && ws.side2 != nullptr;
    cudaStream_t snf = near_early ? ws.side2 : sn;
    auto launch_near = [&](bool after_event) -> cudaError_t {
        cudaError_t r;
        if (fork && after_event && (r = cudaStreamWaitEvent(snf, ws.ev_p2m, 0)) != cudaSuccess)
            return r;
        if (ws.kev[2] && (r = record_timing(ws.kev[2], snf)) !=
                             cudaSuccess)
            return r;
        launch_p2p<T>(D, leaves, leaf_grid, phi != nullptr, ws, ws.cid + dl.off[D], near, snf);
        if ((r = cudaGetLastError()) != cudaSuccess) return r;
        if (ws.kev[3] && (r = record_timing(ws.kev[3], snf)) !=
                             cudaSuccess)
            return r;
        if (fork && (r = cudaEventRecord(ws.ev_near, snf)) != cudaSuccess) return r;
        return cudaSuccess;
    };
    if (nf && near_early) {
        if ((e = cudaStreamWaitEvent(snf, ws.ev_fork, 0)) != cudaSuccess) return e;
        if ((e = launch_near(false)) != cudaSuccess) return e;
    }
    const bool near_late = fork && use_tc && !near_early;
    if (f64 && (e = launch_f64_slice(n, D, (const double*)ws.M, ws, s)) != cudaSuccess) return e;
    if (nf && !near_late && !near_early) {
        if (fork && (e = cudaEventRecord(ws.ev_p2m, s)) != cudaSuccess) return e;
        if ((e = launch_near(true)) != cudaSuccess) return e;
    }
    if (far) {
        for (int l = lmin_p2m - 1; l >= 2; --l) {
            if (use_tc) {
                e = level_cap(n, l) <= kShiftSmallM2M ? launch_shift_small(0, n, D, l, ws, s)
                                                      : launch_m2m_tc(n, D, l, ws, s);
                if (e != cudaSuccess) return e;
                continue;
            }
            if (f64) {
                if ((e = launch_f64_m2m(n, D, l, ws, s)) != cudaSuccess) return e;
                continue;
            }
            if constexpr (sizeof(T) == 4) {
                if ((e = launch_f32_m2m(n, D, l, ws, s)) != cudaSuccess) return e;
            } else {
                int64_t cl = (int64_t)1 << (3 * l);
                int cells = (int)(n < cl ? n : cl);
                int g = (cells + 3) / 4;
                if (g > 152 * 16) g = 152 * 16;
                k_m2m<T><<<g, 128, 4 * P * sizeof(T), s>>>(l, P, ws.ld, ws.linfo, ws.code, ws.cid,
                                                           dl.off[l + 1], (const T*)ws.T_m2m, M);
            }
        }
    }
    if (ev && (e = record_timing(ev[0], s)) != cudaSuccess)
        return e;
    if (far && use_tc) {
        if (fork && (e = cudaStreamWaitEvent(s, ws.ev_items, 0)) != cudaSuccess) return e;
        // L2L down to level D - l2p_levels + 1; the leaves' L2P evaluates the
        // own M2L sums of the leaf and its parent and the complete expansion
        // of the ancestor above them itself (direct mode: no L2L at all)
        if ((e = launch_m2l_tc_run(n, D, ws, direct ? 2 : D + 1 - l2p_levels, split_last, s,
                                   near_late ? ws.ev_p2m : nullptr)) != cudaSuccess)
            return e;
        if (nf && near_late && (e = launch_near(true)) != cudaSuccess) return e;
    } else if (f64) {
        if (pairs_simt && fork && (e = cudaStreamWaitEvent(s, ws.ev_items, 0)) != cudaSuccess)
            return e;
        if (ws.kev[0] && (e = record_timing(ws.kev[0], s)) != cudaSuccess) return e;
        const int64_t tb = target_cells_bound(n, D), step = f64_batched ? ws.f64_batch : tb;
        for (int64_t t0 = 0; t0 < tb; t0 += step) {
            const int b0 = (int)t0, b1 = f64_batched ? (int)(t0 + step) : kAllTargets;
            if (f64_batched && (e = launch_m2l_pairs_worklist(n, D, ws, s, b0, b1)) != cudaSuccess)
                return e;
            if ((e = launch_f64_m2l(ws, s)) != cudaSuccess) return e;
            if (!f64_batched && ws.kev[1] && (e = record_timing(ws.kev[1], s)) != cudaSuccess)
                return e;
            if ((e = launch_m2l_pairs_reduce(n, D, ws, ws.ld, s, b0, b1)) != cudaSuccess) return e;
        }
        if (f64_batched && ws.kev[1] && (e = record_timing(ws.kev[1], s)) != cudaSuccess) return e;
        for (int l = 3; l <= D; ++l)
            if ((e = launch_f64_l2l(n, D, l, ws, s)) != cudaSuccess) return e;
    } else if (pairs_simt) {
        if (fork && (e = cudaStreamWaitEvent(s, ws.ev_items, 0)) != cudaSuccess) return e;
        // M2L products of the work list, the per-target sums, L2L down to
        // the leaves (their L2P evaluates their own expansion)
        if ((e = launch_m2l_pairs_simt(n, D, ws, direct ? 2 : D, s)) != cudaSuccess) return e;
    } else if (far) {
        if (ws.kev[0] && (e = record_timing(ws.kev[0], s)) !=
                             cudaSuccess)
            return e;
        for (int l = 2; l <= D; ++l) {
            if constexpr (sizeof(T) == 4) {
                if ((e = launch_f32_tiles(n, D, l, ws, s)) != cudaSuccess) return e;
            } else {
                int64_t cl = (int64_t)1 << (3 * l);
                int cells = (int)(n < cl ? n : cl);
                dim3 grid((cells + kNT - 1) / kNT + 8, (P + kRT - 1) / kRT);
                k_m2l_simt<T><<<grid, 256, 0, s>>>(l, P, ws.ld, ws.linfo, ws.code, ws.cid, dl.off[l],
                                                   l >= 3 ? dl.off[l - 1] : 0, M, L,
                                                   (const T*)ws.T_m2l, (const T*)ws.T_l2l);
            }
        }
        if (ws.kev[1] && (e = record_timing(ws.kev[1], s)) !=
                             cudaSuccess)
            return e;
    }
    if (ev && (e = record_timing(ev[1], s)) != cudaSuccess)
        return e;
    if (fork && (e = cudaStreamWaitEvent(s, ws.ev_near, 0)) != cudaSuccess) return e;
    if (direct)
        k_l2p_anc<T><<<leaf_grid, kNfThreads, 0, s>>>(
            n, D, 2, p, ws.ld, ws.root, ws.linfo, ws.code, ws.cid,
            (const typename Ion<T>::rec*)ws.sorted, ws.perm, ws.cstart, ws.ccount, L,
            nf ? near : nullptr, E, phi);
    else if (far && sizeof(T) == 8 && n >= kL2pSlotIons)
        e = launch_pdl(phi ? k_l2p_f64<true> : k_l2p_f64<false>,
                       dim3((unsigned)((n + kSlotWindow - 1) / kSlotWindow)), dim3(kSlotThreads),
                       l2p_f64_smem(P), s, n, D, p, ws.ld, l2p_f64_leaves(P), (const RootCube*)ws.root,
                       (const int32_t*)ws.leaf_of, (const int32_t*)ws.cstart,
                       (const int32_t*)ws.ccount, (const Ion<double>::rec*)ws.sorted,
                       (const int32_t*)ws.perm, (const double*)ws.L,
                       (const double*)(nf ? ws.near : nullptr), E, phi);
    else if (far && sizeof(T) == 4 && p <= 15) {
        const int G = !alone || n >= kL2pF32Ions ? 1 : 4, w = l2p_f32_window(G);
        e = launch_pdl(G == 1 ? k_l2p_f32<1> : k_l2p_f32<4>, dim3((unsigned)((n + w - 1) / w)),
                       dim3(l2p_f32_threads(G)), l2p_f32_smem(P, G), s, n, D, p, ws.ld, l2p_levels,
                       l2p_f32_exps(P, G), (const RootCube*)ws.root, (const uint32_t*)ws.code,
                       (const int32_t*)ws.cid, (const int32_t*)ws.leaf_of, (const int32_t*)ws.cstart,
                       (const int32_t*)ws.ccount, (const Ion<float>::rec*)ws.sorted,
                       (const int32_t*)ws.perm, (const float*)ws.L,
                       (const float*)(nf ? ws.near : nullptr), E, phi);
    }
    else
        e = launch_pdl(p <= 15 ? k_l2p<T, 8> : k_l2p<T, 16>, dim3(leaf_grid), dim3(kL2pThreads),
                       0, s, n, D, p, ws.ld, far,
                       l2p_levels, (const RootCube*)ws.root,
                       (const LevelInfo*)ws.linfo, (const uint32_t*)ws.code,
                       (const int32_t*)ws.cid, (const typename Ion<T>::rec*)ws.sorted,
                       (const int32_t*)ws.perm, (const int32_t*)ws.cstart,
                       (const int32_t*)ws.ccount, (const T*)L, (const T*)(nf ? near : nullptr),
                       E, phi);
    if (e != cudaSuccess) return e;
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    if (ev && (e = record_timing(ev[2], s)) != cudaSuccess)
        return e;
    return cudaSuccess;
}

cudaError_t launch_fmm_phased(int64_t n, int D, int phases, Workspace& ws, bool use_tc, double* E,
                              double* phi, cudaStream_t s, cudaEvent_t* ev, bool alone) {
    if (ws.fp64) return run_fmm<double>(n, D, phases, ws, false, E, phi, s, ev, alone);
    return run_fmm<float>(n, D, phases, ws, use_tc, E, phi, s, ev, alone);
}

cudaError_t launch_fmm(int64_t n, int D, int phases, Workspace& ws, bool use_tc, double* E,
                       double* phi, cudaStream_t s) {
    return launch_fmm_phased(n, D, phases, ws, use_tc, E, phi, s, nullptr, true);
}

// M2M into level l (mode 0) or L2L into level l (mode 1) of a small level of
// the tensor-core paths on the CUDA cores (k_shift_rows; FP32 plans).
cudaError_t launch_shift_small(int mode, int64_t n, int D, int l, Workspace& ws, cudaStream_t s) {
    const int P = ws.P;
    const DenseLayout dl = dense_layout(D);
    const unsigned rg = (unsigned)((P + kShRows - 1) / kShRows);
    const int64_t cl = (int64_t)1 << (3 * l);
    const int64_t cells = n < cl ? n : cl;
    if (mode == 0) {
        const int64_t ch = (cells + ShCells<0>::v - 1) / ShCells<0>::v;
        return launch_pdl(k_shift_rows<float, 0>, dim3(rg, (unsigned)(ch < 16 ? ch : 16)),
                          dim3(kShThreads), shift_rows_smem<float, 0>(P), s, l, P, ws.ld,
                          (const LevelInfo*)ws.linfo, (const uint32_t*)ws.code,
                          (const int32_t*)ws.cid, dl.off[l + 1], (const float*)ws.T_m2m,
                          (float*)ws.M, ws.tc_bf16 ? ws.M_pieces : (uint16_t*)nullptr);
    }
    // per octant: runs of 16 children, a few blocks per octant
    const int64_t ch = (cells + ShCells<1>::v * 8 - 1) / (ShCells<1>::v * 8);
    return launch_pdl(k_shift_rows<float, 1>, dim3(rg, 8, (unsigned)(ch < 4 ? (ch > 0 ? ch : 1) : 4)),
                      dim3(kShThreads), shift_rows_smem<float, 1>(P), s, l, P, ws.ld,
                      (const LevelInfo*)ws.linfo, (const uint32_t*)ws.code, (const int32_t*)ws.cid,
                      dl.off[l - 1], (const float*)ws.T_l2l, (float*)ws.L, (uint16_t*)nullptr);
}

// ---------------------------------------------------------------------------
// Interaction counts of the current tree (for algorithmic work accounting).
// ---------------------------------------------------------------------------
__global__ void k_tree_stats(int D, const LevelInfo* linfo, const uint32_t* __restrict__ code,
                             const int32_t* __restrict__ cid, DenseLayout dl,
                             const int32_t* __restrict__ ccount, unsigned long long* st) {
    const int lmin = dl.lmin;
    const int g0 = linfo->gbase[lmin], g1 = linfo->gbase[D + 1];
    unsigned long long m2l = 0, p2p = 0, shifts = 0;
    for (int g = g0 + blockIdx.x * blockDim.x + threadIdx.x; g < g1; g += gridDim.x * blockDim.x) {
        int l = lmin;
        while (l < D && g >= linfo->gbase[l + 1]) ++l;
        int ix, iy, iz;
        demorton3(code[g], ix, iy, iz);
        const int lim = 1 << l;
        if (l >= 2) {
            const int oct = code[g] & 7;
            for (int t = 0; t < 189; ++t) {
                int opi = c_m2l_off[oct][t];
                int sx = ix - (opi / 49 - 3), sy = iy - ((opi / 7) % 7 - 3), sz = iz - (opi % 7 - 3);
                if (sx < 0 || sy < 0 || sz < 0 || sx >= lim || sy >= lim || sz >= lim) continue;
                if (cid[dl.off[l] + morton3(sx, sy, sz)] >= 0) ++m2l;
            }
        }
        if (l >= 3) ++shifts;
        if (l == D) {
            long long cnt = ccount[g], nb = 0;
            for (int dx = -1; dx <= 1; ++dx)
                for (int dy = -1; dy <= 1; ++dy)
                    for (int dz = -1; dz <= 1; ++dz) {
                        int nx = ix + dx, ny = iy + dy, nz = iz + dz;
                        if (nx < 0 || ny < 0 || nz < 0 || nx >= lim || ny >= lim || nz >= lim) continue;
                        int gn = cid[dl.off[D] + morton3(nx, ny, nz)];
                        if (gn >= 0) nb += ccount[gn];
                    }
            p2p += (unsigned long long)(cnt * nb - cnt);
        }
    }
    atomicAdd(&st[0], m2l);
    atomicAdd(&st[1], p2p);
    atomicAdd(&st[2], shifts);
}

cudaError_t launch_tree_stats(int64_t n, int D, Workspace& ws, int64_t* out, cudaStream_t s) {
    cudaError_t e = cudaMemsetAsync(ws.stats, 0, sizeof(unsigned long long) * 8, s);
    if (e != cudaSuccess) return e;
    DenseLayout dl = dense_layout(D);
    k_tree_stats<<<152, 256, 0, s>>>(D, ws.linfo, ws.code, ws.cid, dl, ws.ccount, ws.stats);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    unsigned long long h[3];
    LevelInfo li;
    if ((e = cudaMemcpyAsync(h, ws.stats, sizeof h, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaMemcpyAsync(&li, ws.linfo, sizeof li, cudaMemcpyDeviceToHost, s)) != cudaSuccess) return e;
    if ((e = cudaStreamSynchronize(s)) != cudaSuccess) return e;
    out[0] = n;
    out[1] = D;
    out[2] = li.gbase[D + 1] - li.gbase[D];
    out[3] = D >= 2 ? li.gbase[D + 1] - li.gbase[2] : 0;
    out[4] = (int64_t)h[0];
    out[5] = (int64_t)h[1];
    out[6] = (int64_t)h[2];
    out[7] = (int64_t)h[2];
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// Direct O(N^2) field in FP64 (Eq. hamiltonian), shared-memory source tiles,
// Neumaier-compensated accumulation.
// ---------------------------------------------------------------------------
struct Neu {
    double s = 0, c = 0;
    __device__ __forceinline__ void add(double v) {
        double t = s + v;
        if (fabs(s) >= fabs(v)) c += (s - t) + v;
        else c += (v - t) + s;
        s = t;
    }
    __device__ __forceinline__ double val() const { return s + c; }
};

__global__ void __launch_bounds__(256) k_direct(int64_t n, const double* __restrict__ pos,
                                                const double* __restrict__ q, double* E,
                                                double* phi) {
    __shared__ double4_32a tile[256];
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    double xi = 0, yi = 0, zi = 0;
    if (i < n) { xi = pos[i]; yi = pos[n + i]; zi = pos[2 * n + i]; }
    Neu ax, ay, az, ap;
    for (int64_t t0 = 0; t0 < n; t0 += 256) {
        int64_t j = t0 + threadIdx.x;
        tile[threadIdx.x] = j < n ? make_double4_32a(pos[j], pos[n + j], pos[2 * n + j], q[j])
                                  : make_double4_32a(0, 0, 0, 0);
        __syncthreads();
        int cnt = (int)(n - t0 < 256 ? n - t0 : 256);
        for (int k = 0; k < cnt; ++k) {
            if (t0 + k == i) continue;
            double4_32a o = tile[k];
            double dx = xi - o.x, dy = yi - o.y, dz = zi - o.z;
            double r2 = dx * dx + dy * dy + dz * dz;
            double r = sqrt(r2);
            double ir = 1.0 / r;
            double w = o.w * ir / r2;
            ax.add(w * dx);
            ay.add(w * dy);
            az.add(w * dz);
            ap.add(o.w * ir);
        }
        __syncthreads();
    }
    if (i < n) {
        E[i] = kCoulomb * ax.val();
        E[n + i] = kCoulomb * ay.val();
        E[2 * n + i] = kCoulomb * az.val();
        if (phi) phi[i] = kCoulomb * ap.val();
    }
}

cudaError_t launch_direct(int64_t n, const double* pos, const double* q, double* E, double* phi,
                          cudaStream_t s) {
    int grid = (int)((n + 255) / 256);
    k_direct<<<grid > 0 ? grid : 1, 256, 0, s>>>(n, pos, q, E, phi);
    return cudaGetLastError();
}

cudaError_t upload_harmonic_tables() {
    static HarmTables<double> hd;
    static HarmTables<float> hf;
    static int16_t off[8][189];
    static bool filled = false;
    if (!filled) {
        fill_harm_tables(hd);
        fill_harm_tables(hf);
        host_m2l_offsets(off);
        filled = true;
    }
    cudaError_t e = cudaMemcpyToSymbol(c_tab_d, &hd, sizeof hd);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_tab_f, &hf, sizeof hf);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_tab_d, &hd, sizeof hd);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(g_tab_f, &hf, sizeof hf);
    if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_m2l_off, off, sizeof off);
    const int pmax = (kMaxOrder + 1) * (kMaxOrder + 1);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_p2m<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kP2mIons * pmax * (int)sizeof(double));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_p2m_f64, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kSlotThreads * p2m_f64_stride(pmax) * (int)sizeof(double));
    // (the largest over the orders: fewer leaves above the order where 16 fit)
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_l2p_f32<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_l2p_f32<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 80 * 1024);
    for (auto f : {k_l2p_f64<true>, k_l2p_f64<false>})
        if (e == cudaSuccess)
            e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, 104 * 1024);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_p2m<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kP2mIons * pmax * (int)sizeof(float));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_p2m_anc<double>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kP2mAncIons * pmax * (int)sizeof(double));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_p2m_anc<float>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 kP2mAncIons * pmax * (int)sizeof(float));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_shift_rows<float, 0>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)shift_rows_smem<float, 0>(pmax));
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_shift_rows<float, 1>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)shift_rows_smem<float, 1>(pmax));
    return e;
}

// ---------------------------------------------------------------------------
// Joined ensemble launches (join.cuh) of the FP32 stages of the tensor-core
// and CUDA-core precisions.
// ---------------------------------------------------------------------------
struct P2mJoin {
    template <class... A>
    __device__ __forceinline__ void operator()(const BlockId& b, const A&... a) const { k_p2m_body<float>(b, a...); }
};
struct P2mAncJoin {
    template <class... A>
    __device__ __forceinline__ void operator()(const BlockId& b, const A&... a) const { k_p2m_anc_body<float>(b, a...); }
};
struct ShiftJoin {
    template <class... A>
    __device__ __forceinline__ void operator()(const BlockId& b, const A&... a) const {
        k_shift_rows_body<float, 0>(b, a...);
    }
};
struct P2pJoin {
    template <class... A>
    __device__ __forceinline__ void operator()(const BlockId& b, const A&... a) const { k_p2p_body(b, a...); }
};
struct L2pJoin {
    template <class... A>
    __device__ __forceinline__ void operator()(const BlockId& b, const A&... a) const {
        k_l2p_body<float, 8>(b, a...);
    }
};
struct L2pSlotJoin {  // members take one thread an ion
    template <class... A>
    __device__ __forceinline__ void operator()(const BlockId& b, const A&... a) const {
        k_l2p_f32_body<1>(b, a...);
    }
};

cudaError_t join_fmm(JoinCtx& c) {
    cudaError_t e = join_kernel<P2mJoin, kP2mThreads, 3>(c, k_p2m<float>);
    if (e == cudaSuccess) e = join_kernel<P2mAncJoin, kP2mThreads, 4>(c, k_p2m_anc<float>);
    if (e == cudaSuccess) e = join_kernel<ShiftJoin, kShThreads, 3>(c, k_shift_rows<float, 0>);
    if (e == cudaSuccess) e = join_kernel<P2pJoin, kNfThreads, 1>(c, k_p2p);
    if (e == cudaSuccess) e = join_kernel<L2pJoin, kL2pThreads, 7>(c, k_l2p<float, 8>);
    if (e == cudaSuccess) e = join_kernel<L2pSlotJoin, l2p_f32_threads(1), 6>(c, k_l2p_f32<1>);
    return e;
}

}  // namespace pt
