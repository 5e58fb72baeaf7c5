// mh.cu -- Metropolis-Hastings potential-energy initialisation of a crystal
// (Sec. 4: starting from an equilibrium, ions are displaced one after the
// other by a random distance below dx in a random direction; a move is kept
// if the crystal's potential energy falls, or else with probability
// exp(-dE / (k_B T)); one scan visits every ion once).
//
// Potential energy: the rotating-frame one at the state's time (Eq. pe_rot
// with the wall phase (c, s) = (cos w_r t, sin w_r t) given by the caller):
// per ion U(x) = q k_z (2 z^2 - x^2 - y^2)/4 + (q B w_r - m w_r^2)(x^2 + y^2)/2
// + q k_z delta (x_r^2 - y_r^2)/4, plus the Coulomb pair energy, so moving
// ion i from a to b changes it by
//   dE = (U(b) - U(a)) + k_e q_i sum_{j != i} q_j (1/|b - x_j| - 1/|a - x_j|).
//
// Random numbers (rng.cuh's Philox, the photon-kick stream with beam field
// 0xFF, the scan in place of the step): slot 0 words (0,1) -> the distance
// fraction, (2,3) -> the accept uniform; slots 1, 2, ... -> (v1, v2) pairs of
// Marsaglia's disc pick of the direction.  The distance depends on |b - a|
// only: the proposal is symmetric.
//
// The chain is sequential, but only through the moves that were kept: a
// batch of kMhBatch consecutive moves is summed against the positions at its
// start on the whole GPU, together with what each kept move j of the batch
// adds to the energy change of each later one k,
//   C_jk = k_e q_k q_j [(1/|b_k - b_j| - 1/|a_k - b_j|) - (1/|b_k - a_j| - 1/|a_k - a_j|)],
// and one warp then takes the decisions in order, adding row j of C to the
// later ones whenever move j is kept.  Between two kept moves nothing
// changes, so it goes from one kept move to the next.  A batch with a move too
// close to its threshold for the rounding of these sums is decided move after
// move, each summed at its turn.  Three kernels:
//   k_mh_draw    once per scan: every ion's proposal (an ion moves once a
//                scan, so its own position is the scan's start's), U(b) - U(a)
//                and the window of dE around -k_B T ln u outside of which the
//                decision is certain without the exponential (inside, the
//                batch is decided move after move);
//   k_mh_sums    per batch: the sums and C (FP64, bound by the FP64 units:
//                2 rsqrt per pair);
//   k_mh_decide  per batch: one block, the decisions by its first warp.
// 1,000 ions: 4.9 us a move by one cluster of 8 CTAs (a cluster barrier per
// move, FP64 on 8 SMs) before, 0.3 us now.
// Compiled with -fmad=false like the push, so the proposal and U are the
// literal IEEE sequence; the pair sums (explicit fma, rsqrt, their order)
// differ from the sequential 1/sqrt sum only in the last bits of dE.
#include <cuda_runtime.h>

#include <algorithm>

#include "internal.h"
#include "rng.cuh"

namespace pt {

namespace {

constexpr int kMhSumThreads = 128;
constexpr int kMhDecideThreads = 1024;

__device__ __forceinline__ double mh_u_ext(const MhParams& mp, double qi, double x, double y,
                                           double z) {
    const double xr = mp.c * x - mp.s * y, yr = mp.s * x + mp.c * y, r2 = x * x + y * y;
    return 0.25 * qi * mp.kz * (2.0 * z * z - r2) + 0.5 * (qi * mp.B * mp.wr - mp.m * mp.wr * mp.wr) * r2 +
           0.25 * qi * mp.kz * mp.delta * (xr * xr - yr * yr);
}

__global__ void __launch_bounds__(128) k_mh_draw(int64_t n, const double* __restrict__ x,
                                                 const double* __restrict__ y,
                                                 const double* __restrict__ z,
                                                 const double* __restrict__ q, MhParams mp,
                                                 uint64_t scan, double* prop) {
    pdl_wait();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    uint32_t w[4];
    philox4x32_10((uint32_t)i, 0xFFu, (uint32_t)scan, (uint32_t)(scan >> 32), (uint32_t)mp.seed,
                  (uint32_t)(mp.seed >> 32), w);
    const double r = mp.dx * u01(w[0], w[1]);
    const double u = u01(w[2], w[3]);
    double v1 = 0.0, v2 = 0.0, ss = 0.0;
    for (uint32_t slot = 1; slot <= (uint32_t)kMaxTries; ++slot) {
        philox4x32_10((uint32_t)i, 0xFFu | (slot << 8), (uint32_t)scan, (uint32_t)(scan >> 32),
                      (uint32_t)mp.seed, (uint32_t)(mp.seed >> 32), w);
        v1 = 2.0 * u01(w[0], w[1]) - 1.0;
        v2 = 2.0 * u01(w[2], w[3]) - 1.0;
        ss = v1 * v1 + v2 * v2;
        if (ss < 1.0) break;
    }
    const double f = 2.0 * sqrt(1.0 - ss);
    const double ax = x[i], ay = y[i], az = z[i];
    const double bx = ax + r * (v1 * f), by = ay + r * (v2 * f), bz = az + r * (1.0 - 2.0 * ss);
    // dE < -k_B T ln u keeps the move; within 1e-9 (k_B T + that) of it, or
    // with u = 0, the exponential decides
    const double kt = mp.kb * mp.temp;
    double lo = -INFINITY, hi = INFINITY;
    if (u > 0.0) {
        const double thr = -kt * log(u), margin = 1e-9 * (kt + thr);
        lo = thr - margin;
        hi = thr + margin;
    }
    double* p = prop + i;
    p[0] = bx;
    p[n] = by;
    p[2 * n] = bz;
    p[3 * n] = mh_u_ext(mp, q[i], bx, by, bz) - mh_u_ext(mp, q[i], ax, ay, az);
    p[4 * n] = lo;
    p[5 * n] = hi;
    p[6 * n] = u;
}

__device__ __forceinline__ double mh_inv(double dx, double dy, double dz) {
    return rsqrt(fma(dz, dz, fma(dy, dy, dx * dx)));
}

// the high word of a magnitude: ordered as the magnitudes are
__device__ __forceinline__ unsigned mh_high(double v) {
    return (unsigned)__double2hiint(v) & 0x7fffffffu;
}

// blocks [0, sum_blocks): a warp per (move, source range); the rest: a
// thread per (j, k) of C, j < k, and the largest |C| (its high word) into *top
__global__ void __launch_bounds__(kMhSumThreads) k_mh_sums(
    int64_t n, int64_t i0, int nb, int chunks, int64_t per, int sum_blocks,
    const double* __restrict__ x, const double* __restrict__ y, const double* __restrict__ z,
    const double* __restrict__ q, double ke, const double* __restrict__ prop, double* part, double* C,
    unsigned* top) {
    pdl_wait();
    const int lane = threadIdx.x & 31;
    if ((int)blockIdx.x < sum_blocks) {
        const int u = (int)((blockIdx.x * kMhSumThreads + threadIdx.x) >> 5);
        const int k = u / chunks, c = u % chunks;
        if (k >= nb) return;
        const int64_t i = i0 + k, j1 = min(n, (c + 1) * per);
        const double ax = x[i], ay = y[i], az = z[i];
        const double bx = prop[i], by = prop[n + i], bz = prop[2 * n + i];
        double s = 0.0;
        for (int64_t j = c * per + lane; j < j1; j += 32) {
            const double xj = x[j], yj = y[j], zj = z[j];
            const double ib = mh_inv(bx - xj, by - yj, bz - zj), ia = mh_inv(ax - xj, ay - yj, az - zj);
            if (j != i) s = fma(q[j], ib - ia, s);
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if (lane == 0) part[k * chunks + c] = s;
        return;
    }
    const int e = ((int)blockIdx.x - sum_blocks) * kMhSumThreads + threadIdx.x;
    const int j = e / nb, k = e % nb;
    double c = 0.0;
    if (j < nb && k > j) {
        const int64_t ij = i0 + j, ik = i0 + k;
        const double ajx = x[ij], ajy = y[ij], ajz = z[ij], akx = x[ik], aky = y[ik], akz = z[ik];
        const double bjx = prop[ij], bjy = prop[n + ij], bjz = prop[2 * n + ij];
        const double bkx = prop[ik], bky = prop[n + ik], bkz = prop[2 * n + ik];
        const double after = mh_inv(bkx - bjx, bky - bjy, bkz - bjz) - mh_inv(akx - bjx, aky - bjy, akz - bjz);
        const double before = mh_inv(bkx - ajx, bky - ajy, bkz - ajz) - mh_inv(akx - ajx, aky - ajy, akz - ajz);
        c = ke * q[ik] * (q[ij] * (after - before));
        C[j * kMhBatch + k] = c;
    }
    const unsigned t = __reduce_max_sync(0xffffffffu, mh_high(c));
    if (lane == 0 && t > 0u) atomicMax(top, t);
}

// The decisions of a batch, each move summed at its turn by the whole block:
// the moves kept so far (marked in kept) are made.
__device__ __noinline__ void mh_one_by_one(int64_t n, int64_t i0, int nb, const double* x,
                                           const double* y, const double* z,
                                           const double* __restrict__ q, const MhParams& mp,
                                           const double* __restrict__ prop, unsigned* kept,
                                           double* red, unsigned long long* acc_out, double* de_out) {
    const int tid = threadIdx.x;
    if (tid < kMhBatch / 32) kept[tid] = 0u;
    __syncthreads();
    for (int j = 0; j < nb; ++j) {
        const double ax = x[i0 + j], ay = y[i0 + j], az = z[i0 + j];
        const double bx = prop[i0 + j], by = prop[n + i0 + j], bz = prop[2 * n + i0 + j];
        double s = 0.0;
        for (int64_t c = tid; c < n; c += kMhDecideThreads) {
            const int64_t k = c - i0;
            if (k == j) continue;
            const bool made = k >= 0 && k < j && ((kept[k >> 5] >> (k & 31)) & 1u);
            const double xc = made ? prop[c] : x[c], yc = made ? prop[n + c] : y[c],
                         zc = made ? prop[2 * n + c] : z[c];
            s = fma(q[c], mh_inv(bx - xc, by - yc, bz - zc) - mh_inv(ax - xc, ay - yc, az - zc), s);
        }
        for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
        if ((tid & 31) == 0) red[tid >> 5] = s;
        __syncthreads();
        if (tid == 0) {
            double sum = 0.0;
            for (int w = 0; w < kMhDecideThreads / 32; ++w) sum += red[w];
            const int64_t i = i0 + j;
            const double dE = prop[3 * n + i] + mp.ke * q[i] * sum;
            if (dE < 0.0 || prop[6 * n + i] < pt_exp(-dE / (mp.kb * mp.temp))) {
                kept[j >> 5] |= 1u << (j & 31);
                ++*acc_out;
                *de_out += dE;
            }
        }
        __syncthreads();
    }
}

// The decisions of a batch.  Lane l of warp 0 holds moves l + 32 m.
// With S the largest of the batch's energy changes and of the terms C, a sum
// of them is within 2^-38 S of the sum without rounding.  A batch with a move
// that close to its threshold is decided one by one: at the energies of a
// crystal (S = 1e3 k_B T) one in 1e6, and those where ions coincide or all
// but (S infinite: infinite terms do not cancel).
__global__ void __launch_bounds__(kMhDecideThreads) k_mh_decide(
    int64_t n, int64_t i0, int nb, int chunks, double* x, double* y, double* z,
    const double* __restrict__ q, const __grid_constant__ MhParams mp,
    const double* __restrict__ prop, const double* __restrict__ part,
    const double* __restrict__ C, unsigned* top, unsigned long long* acc_out, double* de_out) {
    extern __shared__ double sC[];  // [nb][kMhBatch]
    __shared__ double s_sum[kMhBatch], s_red[kMhDecideThreads / 32];
    __shared__ unsigned s_kept[kMhBatch / 32];
    __shared__ bool s_anew;
    pdl_wait();
    const int tid = threadIdx.x, lane = tid & 31;
    const unsigned top_c = *top;
#pragma unroll 8
    for (int e = tid; e < nb * kMhBatch; e += kMhDecideThreads)
        if (e % kMhBatch > e / kMhBatch) sC[e] = C[e];
    if (tid < nb) {
        double s = 0.0;
        for (int c = 0; c < chunks; ++c) s += part[tid * chunks + c];
        s_sum[tid] = s;
    }
    __syncthreads();
    if (tid < 32) {
        constexpr int NM = kMhBatch / 32;
        double E[NM], lo[NM], hi[NM];  // dE with the moves kept so far
        unsigned t = top_c;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int k = lane + 32 * m;
            E[m] = k < nb ? prop[3 * n + i0 + k] + mp.ke * q[i0 + k] * s_sum[k] : 0.0;
            t = max(t, mh_high(E[m]));
        }
        t = __reduce_max_sync(0xffffffffu, t);
        const double slack = t < 0x7ff00000u ? 0x1p-38 * __hiloint2double((int)t, -1) : (double)INFINITY;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            const int64_t i = i0 + lane + 32 * m;
            const bool live = lane + 32 * m < nb;
            lo[m] = live ? prop[4 * n + i] - slack : 0.0;
            hi[m] = live ? prop[5 * n + i] + slack : 0.0;
        }
        unsigned long long acc = 0;
        double de_sum = *de_out;
        bool anew = false;
#pragma unroll
        for (int m = 0; m < NM; ++m) {
            // the first undecided move of the group that may be kept: the
            // undecided ones before it are not (nothing changed since)
            const int nl = nb - 32 * m;  // moves left, this group's first
            unsigned left = nl >= 32 ? 0xffffffffu : nl > 0 ? (1u << nl) - 1u : 0u, kept = 0;
            while (left && !anew) {
                const unsigned may = __ballot_sync(0xffffffffu, !(E[m] > hi[m])) & left;
                const unsigned sure = __ballot_sync(0xffffffffu, E[m] < lo[m]);
                if (!may) break;
                const int l = __ffs(may) - 1, j = l + 32 * m;
                left = l == 31 ? 0u : left & (0xffffffffu << (l + 1));
                if (!((sure >> l) & 1u)) {
                    anew = true;
                    break;
                }
                kept |= 1u << l;
                ++acc;
                de_sum += __shfl_sync(0xffffffffu, E[m], l);
                // (the columns up to j are decided, those from nb on are no moves:
                // what is added there is unused)
                const double* row = sC + j * kMhBatch + lane;
#pragma unroll
                for (int mm = m; mm < NM; ++mm) E[mm] += row[32 * mm];
            }
            if (lane == 0) s_kept[m] = kept;
        }
        if (lane == 0) {
            s_anew = anew;
            *top = 0u;  // for the next batch
            if (!anew) {
                *acc_out += acc;
                *de_out = de_sum;
            }
        }
    }
    __syncthreads();
    if (s_anew) mh_one_by_one(n, i0, nb, x, y, z, q, mp, prop, s_kept, s_red, acc_out, de_out);
    if (tid < nb && ((s_kept[tid >> 5] >> (tid & 31)) & 1u)) {
        const int64_t i = i0 + tid;
        x[i] = prop[i];
        y[i] = prop[n + i];
        z[i] = prop[2 * n + i];
    }
}

}  // namespace

cudaError_t launch_mh_scans(int64_t n, double* x, double* y, double* z, const double* q,
                            const MhParams& mp, int64_t scan0, int64_t n_scans,
                            unsigned long long* acc_out, double* de_out, double* scratch, int sms,
                            cudaStream_t s) {
    double* prop = scratch;
    double* part = prop + (size_t)kMhProp * n;
    double* C = part + kMhBatch * kMhMaxChunks;
    unsigned* top = reinterpret_cast<unsigned*>(C + kMhBatch * kMhBatch);
    const int smem = (int)sizeof(double) * kMhBatch * kMhBatch;
    cudaError_t e = cudaFuncSetAttribute(k_mh_decide, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e == cudaSuccess) e = cudaMemsetAsync(acc_out, 0, sizeof *acc_out, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(de_out, 0, sizeof *de_out, s);
    if (e == cudaSuccess) e = cudaMemsetAsync(top, 0, sizeof *top, s);
    // source ranges of whole warps' worth, about eight warps per SM over the batch
    const int64_t want = (sms * 8 + kMhBatch - 1) / kMhBatch;
    int64_t chunks = std::min<int64_t>(std::min<int64_t>(want, kMhMaxChunks), (n + 31) / 32);
    const int64_t per = ((n + chunks - 1) / chunks + 31) / 32 * 32;
    chunks = (n + per - 1) / per;
    for (int64_t sc = 0; sc < n_scans && e == cudaSuccess; ++sc) {
        e = launch_pdl(k_mh_draw, dim3((unsigned)((n + 127) / 128)), dim3(128), 0, s, n, (const double*)x,
                       (const double*)y, (const double*)z, q, mp, (uint64_t)(scan0 + sc), prop);
        for (int64_t i0 = 0; i0 < n && e == cudaSuccess; i0 += kMhBatch) {
            const int nb = (int)std::min<int64_t>(kMhBatch, n - i0);
            const int wpb = kMhSumThreads / 32;
            const int sb = (int)((nb * chunks + wpb - 1) / wpb);
            const int cb = (nb * nb + kMhSumThreads - 1) / kMhSumThreads;
            e = launch_pdl(k_mh_sums, dim3((unsigned)(sb + cb)), dim3(kMhSumThreads), 0, s, n, i0, nb,
                           (int)chunks, per, sb, (const double*)x, (const double*)y, (const double*)z,
                           q, mp.ke, (const double*)prop, part, C, top);
            if (e == cudaSuccess)
                e = launch_pdl(k_mh_decide, dim3(1), dim3(kMhDecideThreads), (size_t)smem, s, n, i0, nb,
                               (int)chunks, x, y, z, q, mp, (const double*)prop, (const double*)part,
                               (const double*)C, top, acc_out, de_out);
        }
    }
    return e;
}

}  // namespace pt
