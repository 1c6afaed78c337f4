// Device body of the series accumulate (arxiv 2307.03968 eqs. 20-22: x_j = y -
// D^{-1} z) for one leaf, shared by the leaf-update kernel (k_solve.cu) and the
// one-launch solve (k_persist.cu).  Its vector pointers carry no __restrict__:
// in the one-launch solve they are written by other CTAs between phases.
#pragma once

#include "k_common.cuh"

namespace hm {
namespace {

using namespace kc;

// The leaf product w = D_i^{-1} z for RB right-hand sides of one leaf, by a CTA of 256
// threads: rows rc0 .. rc0 + 63, then every rcs rows on.  D_i^{-1} is column-major np x np
// (np = padded leaf length, zero padded); zs[q * np + j] holds right-hand side q's leaf
// vector, part 8 * RB * 64 entries, both in the caller's shared memory.  Warp w takes every
// 8th column, a lane two rows; the warps' sums are added in warp order and given to
// emit(q, row, sum).
template <class T, int RB, class Emit>
__device__ __forceinline__ void leaf_product(const typename CT<T>::C *__restrict__ Di, int np, int rc0, int rcs,
                                             const typename CT<T>::C *zs, typename CT<T>::C *part, Emit emit)
{
    using C = typename CT<T>::C;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int rc = rc0; rc < np; rc += rcs) {
        const int i = rc + 2 * lane;
        C a0[RB], a1[RB];
#pragma unroll
        for (int q = 0; q < RB; ++q) a0[q] = a1[q] = czero(C());
        if (i < np)
#pragma unroll 4
            for (int j = w; j < np; j += 8) {
                const Pair<T> d = RB == 1 ? ld_stream(Di + (int64_t)j * np + i) : ld_cached(Di + (int64_t)j * np + i);
#pragma unroll
                for (int q = 0; q < RB; ++q) {
                    const C zj = zs[q * np + j];
                    cfma(a0[q], d.a, zj);
                    cfma(a1[q], d.b, zj);
                }
            }
#pragma unroll
        for (int q = 0; q < RB; ++q) {
            part[(w * RB + q) * 64 + 2 * lane] = a0[q];
            part[(w * RB + q) * 64 + 2 * lane + 1] = a1[q];
        }
        __syncthreads();
        for (int e = tid; e < RB * 64; e += 256) {
            const int q = e >> 6, t = e & 63;
            if (rc + t < np) {
                C s = part[q * 64 + t];
#pragma unroll
                for (int v = 1; v < 8; ++v) s = cadd(s, part[(v * RB + q) * 64 + t]);
                emit(q, rc + t, s);
            }
        }
        __syncthreads();
    }
}

// Per leaf and right-hand side (zs: np entries, part: 8 x 64 entries of the caller's shared
// memory):  w = D_i^{-1} zin_i ;  out_i = y ? y_i - w : w ;  zin_i = 0 if zero_in.
template <class T>
__device__ __forceinline__ void leaf_update_leaf(int leaf, int r, const int32_t *__restrict__ pleaf_off,
                                                 const int64_t *__restrict__ dinv_off,
                                                 const typename CT<T>::C *__restrict__ dinv,
                                                 const typename CT<T>::C *y, typename CT<T>::C *zin,
                                                 typename CT<T>::C *out, int64_t ld, int zero_in,
                                                 typename CT<T>::C *zs, typename CT<T>::C *part)
{
    using C = typename CT<T>::C;
    const int o = pleaf_off[leaf], np = pleaf_off[leaf + 1] - o;
    C *zr = zin + r * ld + o;
    for (int j = threadIdx.x; j < np; j += blockDim.x) zs[j] = zr[j];
    __syncthreads();
    if (zero_in)
        for (int j = threadIdx.x; j < np; j += blockDim.x) zr[j] = czero(C());
    const int64_t g = r * ld + o;
    leaf_product<T, 1>(dinv + dinv_off[leaf], np, 0, 64, zs, part,
                       [&](int, int i, C s) { out[g + i] = y ? csub(y[g + i], s) : s; });
}

} // namespace
} // namespace hm
