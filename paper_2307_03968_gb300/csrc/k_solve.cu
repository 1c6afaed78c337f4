// Device kernels of the power-series solve (arxiv 2307.03968 §IV, eqs. 12-22).
//
//  (the block product is in k_product.cu, the FP64-class residual in k_residual.cu)
//  k_leaf_update   per leaf: out = y - D_i^{-1} z_i (the series accumulate of
//                  x_j = y - D^{-1} M x_{j-1}), or out = D_i^{-1} z_i; clears z.
//  helpers         permutation in/out, residual, finiteness check.
#include "k_solve_dev.cuh"

#include <cuda_runtime.h>

namespace hm {
namespace {

using namespace kc;

// The leaf passes: a CTA per leaf (blockIdx.x), group of RB right-hand sides (blockIdx.y)
// and, where the leaves are few and long, row chunk (blockIdx.z; leaf_grid gives the
// split and the reasons).

// the leaf's vectors of RB right-hand sides (nr of them given, zero past them) into zs, all
// loads before the first store, then cleared if asked
template <int RB, class C>
__device__ __forceinline__ void leaf_vectors(C *z, int64_t ld, int np, int nr, int clear, C *zs)
{
    for (int j = threadIdx.x; j < np; j += 256) {
        C v[RB];
#pragma unroll
        for (int q = 0; q < RB; ++q) v[q] = q < nr ? z[q * ld + j] : czero(C());
#pragma unroll
        for (int q = 0; q < RB; ++q) zs[q * np + j] = v[q];
    }
    __syncthreads();
    if (clear)
        for (int j = threadIdx.x; j < np; j += 256)
#pragma unroll
            for (int q = 0; q < RB; ++q)
                if (q < nr) z[q * ld + j] = czero(C());
}

// out = y ? y - D_i^{-1} zin_i : D_i^{-1} zin_i; zin_i cleared if zero_in (one row chunk only)
template <class T, int RB>
__global__ void __launch_bounds__(256)
k_leaf_update(const int32_t *__restrict__ pleaf_off, const int64_t *__restrict__ dinv_off,
              const typename CT<T>::C *__restrict__ dinv, const typename CT<T>::C *y,
              typename CT<T>::C *zin, typename CT<T>::C *out, int64_t ld, int nrhs, int zero_in)
{
    using C = typename CT<T>::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ C part[8 * RB * 64];
    C *zs = reinterpret_cast<C *>(smem_raw);
    const int leaf = blockIdx.x, r0 = blockIdx.y * RB, nr = min(RB, nrhs - r0);
    const int o = pleaf_off[leaf], np = pleaf_off[leaf + 1] - o;
    leaf_vectors<RB>(zin + (int64_t)r0 * ld + o, ld, np, nr, zero_in, zs);
    leaf_product<T, RB>(dinv + dinv_off[leaf], np, 64 * blockIdx.z, 64 * gridDim.z, zs, part, [&](int q, int i, C s) {
        if (q >= nr) return;
        const int64_t g = (int64_t)(r0 + q) * ld + o + i;
        out[g] = y ? csub(y[g], s) : s;
    });
}

// acc += D x for the complex64 self blocks (column-major, like D^{-1}), with
// accumulation in precision A (float or double)
template <class A>
__global__ void __launch_bounds__(256)
k_apply_self(const int32_t *__restrict__ pleaf_off, const int64_t *__restrict__ off,
             const float2 *__restrict__ self, const float2 *__restrict__ x, typename CT<A>::C *acc, int64_t ld)
{
    using CA = typename CT<A>::C;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    CA *xs = reinterpret_cast<CA *>(smem_raw);
    __shared__ CA part[8][64];
    const int leaf = blockIdx.x, r = blockIdx.y;
    const int o = pleaf_off[leaf], np = pleaf_off[leaf + 1] - o;
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
    for (int j = tid; j < np; j += blockDim.x) xs[j] = conv<CA>(x[r * ld + o + j]);
    __syncthreads();
    const float2 *S = self + off[leaf];
    for (int rc = 0; rc < np; rc += 64) {
        const int i = rc + 2 * lane;
        CA a0 = czero(CA()), a1 = czero(CA());
        if (i < np)
            for (int j = w; j < np; j += 8) {
                Pair<float> d = ld_stream(S + (int64_t)j * np + i);
                cfma(a0, conv<CA>(d.a), xs[j]);
                cfma(a1, conv<CA>(d.b), xs[j]);
            }
        part[w][2 * lane] = a0;
        part[w][2 * lane + 1] = a1;
        __syncthreads();
        if (tid < 64 && rc + tid < np) {
            CA s = part[0][tid];
#pragma unroll
            for (int q = 1; q < 8; ++q) s = cadd(s, part[q][tid]);
            const int64_t g = r * ld + o + rc + tid;
            acc[g] = cadd(acc[g], s);
        }
        __syncthreads();
    }
}

template <class C>
__global__ void k_permute_in(const C *__restrict__ b, int64_t ldb, C *__restrict__ xt, int64_t pN,
                             const int32_t *__restrict__ pperm, int nrhs)
{
    const int64_t total = pN * nrhs;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / pN, p = t - r * pN;
        const int32_t src = pperm[p];
        xt[t] = src >= 0 ? b[r * ldb + src] : czero(C());
    }
}

// complex64: the leaf's rows of bt = P b (0 at pads) and y = D_i^{-1} bt_i (the first step
// of the series, eq. 12 applied to the permuted right-hand side)
template <int RB>
__global__ void __launch_bounds__(256)
k_permute_leaf(const int32_t *__restrict__ pleaf_off, const int64_t *__restrict__ dinv_off,
               const float2 *__restrict__ dinv, const int32_t *__restrict__ pperm, const float2 *__restrict__ b,
               int64_t ldb, float2 *bt, float2 *y, int64_t pN, int nrhs)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float2 part[8 * RB * 64];
    float2 *zs = reinterpret_cast<float2 *>(smem_raw);
    const int leaf = blockIdx.x, r0 = blockIdx.y * RB, nr = min(RB, nrhs - r0);
    const int o = pleaf_off[leaf], np = pleaf_off[leaf + 1] - o;
    for (int j = threadIdx.x; j < np; j += 256) {
        const int32_t src = pperm[o + j];
        float2 v[RB];
#pragma unroll
        for (int q = 0; q < RB; ++q)
            v[q] = src >= 0 && q < nr ? b[(int64_t)(r0 + q) * ldb + src] : make_float2(0.f, 0.f);
#pragma unroll
        for (int q = 0; q < RB; ++q) {
            zs[q * np + j] = v[q];
            if (blockIdx.z == 0 && q < nr) bt[(int64_t)(r0 + q) * pN + o + j] = v[q];
        }
    }
    __syncthreads();
    leaf_product<float, RB>(dinv + dinv_off[leaf], np, 64 * blockIdx.z, 64 * gridDim.z, zs, part,
                            [&](int q, int i, float2 s) {
                                if (q < nr) y[(int64_t)(r0 + q) * pN + o + i] = s;
                            });
}

template <class C>
__global__ void k_permute_out(const C *__restrict__ xt, int64_t pN, C *__restrict__ x, int64_t ldx,
                              const int32_t *__restrict__ pperm, int nrhs)
{
    const int64_t total = pN * nrhs;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = t / pN, p = t - r * pN;
        const int32_t dst = pperm[p];
        if (dst >= 0) x[r * ldx + dst] = xt[t];
    }
}

template <class C>
__global__ void k_sub(const C *y, const C *w, C *out, int64_t n)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        out[t] = csub(y[t], w[t]);
}

template <class C>
__global__ void k_add(C *x, const C *dx, int64_t n)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        x[t] = cadd(x[t], dx[t]);
}

template <class C>
__global__ void k_check_finite(const C *x, int64_t n, int *status)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x) {
        const C v = x[t];
        if (!isfinite(v.x) || !isfinite(v.y)) {
            atomicCAS(status, 0, (int)HM_ERR_DIVERGED);
            return;
        }
    }
}

// the end of a complex64 solve in one pass: v = xt (+ dx), non-finite v -> HM_ERR_DIVERGED,
// x[r * ldx + pperm[p]] = v (the refinement's add, the check and the un-permutation)
__global__ void k_finish(const float2 *__restrict__ xt, const float2 *__restrict__ dx, int64_t pN, float2 *__restrict__ x,
                         int64_t ldx, const int32_t *__restrict__ pperm, int nrhs, int *status)
{
    const int64_t total = pN * nrhs;
    bool bad = false;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total; t += (int64_t)gridDim.x * blockDim.x) {
        float2 v = xt[t];
        if (dx) v = cadd(v, dx[t]);
        bad |= !isfinite(v.x) || !isfinite(v.y);
        const int64_t r = t / pN, p = t - r * pN;
        const int32_t dst = pperm[p];
        if (dst >= 0) x[r * ldx + dst] = v;
    }
    if (bad) atomicCAS(status, 0, (int)HM_ERR_DIVERGED);
}

// The last series step of a complex64 solve and the end of the solve:
// v = (base ? base_i : 0) + (y_i - D_i^{-1} z_i) (z_i cleared if zero_in), non-finite v ->
// HM_ERR_DIVERGED, x[r * ldx + pperm[p]] = v.
template <int RB>
__global__ void __launch_bounds__(256)
k_leaf_finish(const int32_t *__restrict__ pleaf_off, const int64_t *__restrict__ dinv_off,
              const float2 *__restrict__ dinv, const float2 *__restrict__ y, float2 *z, const float2 *__restrict__ base,
              int64_t pN, int nrhs, float2 *__restrict__ x, int64_t ldx, const int32_t *__restrict__ pperm, int *status,
              int zero_in)
{
    extern __shared__ __align__(16) unsigned char smem_raw[];
    __shared__ float2 part[8 * RB * 64];
    float2 *zs = reinterpret_cast<float2 *>(smem_raw);
    const int leaf = blockIdx.x, r0 = blockIdx.y * RB, nr = min(RB, nrhs - r0);
    const int o = pleaf_off[leaf], np = pleaf_off[leaf + 1] - o;
    leaf_vectors<RB>(z + (int64_t)r0 * pN + o, pN, np, nr, zero_in, zs);
    bool bad = false;
    leaf_product<float, RB>(dinv + dinv_off[leaf], np, 64 * blockIdx.z, 64 * gridDim.z, zs, part,
                            [&](int q, int i, float2 s) {
                                if (q >= nr) return;
                                const int64_t g = (int64_t)(r0 + q) * pN + o + i;
                                float2 v = csub(y[g], s);
                                if (base) v = cadd(v, base[g]);
                                bad |= !isfinite(v.x) || !isfinite(v.y);
                                const int32_t dst = pperm[o + i];
                                if (dst >= 0) x[(int64_t)(r0 + q) * ldx + dst] = v;
                            });
    if (bad) atomicCAS(status, 0, (int)HM_ERR_DIVERGED);
}

__global__ void k_f32_to_f64(const float2 *a, double2 *b, int64_t n)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        b[t] = make_double2(a[t].x, a[t].y);
}

__global__ void k_f64_to_f32(const double2 *a, float2 *b, int64_t n)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < n; t += (int64_t)gridDim.x * blockDim.x)
        b[t] = make_float2((float)a[t].x, (float)a[t].y);
}

int grid_for(int64_t n, int block = 256)
{
    int64_t g = (n + block - 1) / block;
    if (g < 1) g = 1;
    if (g > 4096) g = 4096;
    return (int)g;
}

} // namespace

void launch_permute_in(const void *b, int64_t ldb, void *xt, int64_t pN, const int32_t *pperm, int nrhs,
                       bool fp64, cudaStream_t s)
{
    const int g = grid_for(pN * nrhs);
    if (fp64)
        k_permute_in<double2><<<g, 256, 0, s>>>((const double2 *)b, ldb, (double2 *)xt, pN, pperm, nrhs);
    else
        k_permute_in<float2><<<g, 256, 0, s>>>((const float2 *)b, ldb, (float2 *)xt, pN, pperm, nrhs);
}

void launch_permute_out(const void *xt, int64_t pN, void *x, int64_t ldx, const int32_t *pperm, int nrhs,
                        bool fp64, cudaStream_t s)
{
    const int g = grid_for(pN * nrhs);
    if (fp64)
        k_permute_out<double2><<<g, 256, 0, s>>>((const double2 *)xt, pN, (double2 *)x, ldx, pperm, nrhs);
    else
        k_permute_out<float2><<<g, 256, 0, s>>>((const float2 *)xt, pN, (float2 *)x, ldx, pperm, nrhs);
}

void launch_zero(void *p, size_t bytes, cudaStream_t s) { cudaMemsetAsync(p, 0, bytes, s); }

static int64_t max_padded_leaf(hm_matrix h)
{
    int64_t maxnp = 0;
    for (int64_t i = 0; i < h->n_leaves; ++i) maxnp = std::max<int64_t>(maxnp, h->pleaf_off[i + 1] - h->pleaf_off[i]);
    return maxnp;
}

void launch_apply_self_f32(hm_matrix h, const float2 *x, float2 *acc, int nrhs, cudaStream_t s)
{
    dim3 grid((unsigned)h->n_leaves, (unsigned)nrhs);
    k_apply_self<float><<<grid, 256, max_padded_leaf(h) * sizeof(float2), s>>>(h->d_pleaf_off, h->d_dinv_off,
                                                                              h->d_self32, x, acc, h->pN);
}

// Grid of a leaf pass over nrhs right-hand sides.
//  - Row chunks (chunks > 1): one CTA per leaf and right-hand side leaves the GPU idle when
//    the leaves are few: the 64 leaves of 1,050 unknowns of a 67,200-unknown plate took 0.63 ms
//    a pass on 64 of 152 SMs, 0.11 ms in chunks of 64 rows (their 564 MB of inverses need
//    0.083 ms at the measured copy bandwidth).  Above 8 CTAs an SM there is nothing to gain
//    and the chunks would only re-read z, so the split is for fewer CTAs than that.
//  - RB right-hand sides a CTA: the inverse is read (from L2) once for RB of them, where the
//    pass still has 4 CTAs an SM then: 512 leaves of 60 with 181 right-hand sides take 0.177 ms
//    an update, 0.155 the last one and 0.135 the first, instead of 0.31, 0.52 and 0.29.
struct LeafGrid { dim3 grid; int rb, chunks; size_t maxnp; };
static LeafGrid leaf_grid(hm_matrix h, int nrhs, bool batch)
{
    LeafGrid g;
    g.maxnp = (size_t)std::max<int64_t>(max_padded_leaf(h), 1);
    const int64_t sms = h->num_sms > 0 ? h->num_sms : 1;
    g.chunks = leaf_chunks(h, nrhs);
    g.rb = batch && g.chunks == 1 && g.maxnp <= 256 && h->n_leaves * ((nrhs + 3) / 4) >= 4 * sms ? 4 : 1;
    g.grid = dim3((unsigned)h->n_leaves, (unsigned)((nrhs + g.rb - 1) / g.rb), (unsigned)g.chunks);
    return g;
}

int leaf_chunks(hm_matrix h, int nrhs)
{
    const int64_t maxnp = max_padded_leaf(h), sms = h->num_sms > 0 ? h->num_sms : 1;
    return h->n_leaves * nrhs < 8 * sms ? (int)std::max<int64_t>((maxnp + 63) / 64, 1) : 1;
}

void launch_permute_leaf(hm_matrix h, const float2 *b, int64_t ldb, float2 *bt, float2 *y, int nrhs, cudaStream_t s)
{
    const LeafGrid g = leaf_grid(h, nrhs, true);
    auto go = [&](auto kern) {
        kern<<<g.grid, 256, g.rb * g.maxnp * sizeof(float2), s>>>(h->d_pleaf_off, h->d_dinv_off, h->d_dinv32, h->d_pperm,
                                                                  b, ldb, bt, y, h->pN, nrhs);
    };
    if (g.rb == 4) go(k_permute_leaf<4>);
    else go(k_permute_leaf<1>);
}

void launch_leaf_update(hm_matrix h, const void *y, void *zin, void *out, int nrhs, bool zero_in, bool fp64,
                        cudaStream_t s)
{
    const LeafGrid g = leaf_grid(h, nrhs, !fp64);
    const int clear = zero_in && g.chunks == 1;    // else the row chunks of a leaf read z side by side
    if (fp64) {
        k_leaf_update<double, 1><<<g.grid, 256, g.maxnp * sizeof(double2), s>>>(
            h->d_pleaf_off, h->d_dinv_off, h->d_dinv64, (const double2 *)y, (double2 *)zin, (double2 *)out, h->pN, nrhs,
            clear);
    } else {
        auto go = [&](auto kern) {
            kern<<<g.grid, 256, g.rb * g.maxnp * sizeof(float2), s>>>(h->d_pleaf_off, h->d_dinv_off, h->d_dinv32,
                                                                      (const float2 *)y, (float2 *)zin, (float2 *)out,
                                                                      h->pN, nrhs, clear);
        };
        if (g.rb == 4) go(k_leaf_update<float, 4>);
        else go(k_leaf_update<float, 1>);
    }
    if (zero_in && !clear)
        cudaMemsetAsync(zin, 0, (fp64 ? sizeof(double2) : sizeof(float2)) * (size_t)h->pN * nrhs, s);
}

void launch_sub(const void *y, const void *w, void *out, int64_t n, bool fp64, cudaStream_t s)
{
    const int g = grid_for(n);
    if (fp64) k_sub<double2><<<g, 256, 0, s>>>((const double2 *)y, (const double2 *)w, (double2 *)out, n);
    else k_sub<float2><<<g, 256, 0, s>>>((const float2 *)y, (const float2 *)w, (float2 *)out, n);
}

void launch_add_inplace(void *x, const void *dx, int64_t n, bool fp64, cudaStream_t s)
{
    const int g = grid_for(n);
    if (fp64) k_add<double2><<<g, 256, 0, s>>>((double2 *)x, (const double2 *)dx, n);
    else k_add<float2><<<g, 256, 0, s>>>((float2 *)x, (const float2 *)dx, n);
}

void launch_check_finite(const void *x, int64_t n, bool fp64, int *status, cudaStream_t s)
{
    const int g = grid_for(n);
    if (fp64) k_check_finite<double2><<<g, 256, 0, s>>>((const double2 *)x, n, status);
    else k_check_finite<float2><<<g, 256, 0, s>>>((const float2 *)x, n, status);
}

void launch_leaf_finish(hm_matrix h, const float2 *y, float2 *z, const float2 *base, float2 *x, int64_t ldx, int nrhs,
                        cudaStream_t s)
{
    const LeafGrid g = leaf_grid(h, nrhs, true);
    const int clear = g.chunks == 1;
    auto go = [&](auto kern) {
        kern<<<g.grid, 256, g.rb * g.maxnp * sizeof(float2), s>>>(h->d_pleaf_off, h->d_dinv_off, h->d_dinv32, y, z, base,
                                                                  h->pN, nrhs, x, ldx, h->d_pperm, h->d_status, clear);
    };
    if (g.rb == 4) go(k_leaf_finish<4>);
    else go(k_leaf_finish<1>);
    if (!clear) cudaMemsetAsync(z, 0, sizeof(float2) * (size_t)h->pN * nrhs, s);
}

void launch_finish(const float2 *xt, const float2 *dx, int64_t pN, float2 *x, int64_t ldx, const int32_t *pperm,
                   int nrhs, int *status, cudaStream_t s)
{
    k_finish<<<grid_for(pN * nrhs), 256, 0, s>>>(xt, dx, pN, x, ldx, pperm, nrhs, status);
}

void launch_convert_f32_to_f64(const float2 *a, double2 *b, int64_t n, cudaStream_t s)
{
    k_f32_to_f64<<<grid_for(n), 256, 0, s>>>(a, b, n);
}

void launch_convert_f64_to_f32(const double2 *a, float2 *b, int64_t n, cudaStream_t s)
{
    k_f64_to_f32<<<grid_for(n), 256, 0, s>>>(a, b, n);
}

} // namespace hm
