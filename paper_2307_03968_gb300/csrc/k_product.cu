// Block product z += M x over a list of stored blocks (arxiv 2307.03968 eq. 6
// and eq. 8, with the half storage of §III: every stored block is read once and
// acts on both of its clusters):
//     dense  B (I,J):  z_I += B x_J,            z_J += B^T x_I
//     low rank U V:    z_I += U (V x_J),        z_J += V^T (U^T x_I)
// One warp per block, persistent grid (occupancy x SMs, 8 warps per CTA).  The
// complex64 instantiation is launched with three CTAs per SM (at most 80
// registers a thread), so that 24 warps per SM keep loads in flight.  A lane owns
// two adjacent columns, loaded as one 128-bit streaming load, so column-side sums
// accumulate in registers; row-side sums are warp transpose reductions.  Low-rank
// panels go in chunks of 8 rank rows held in registers, so U^T and V are read
// once.  Results go to z with vector atomics (order-free sums: reproducible to
// FP32 rounding, not bitwise).
#include "k_product_dev.cuh"

namespace hm {
namespace {

using namespace kc;
constexpr int APPLY_WARPS = 8;   // warps per CTA of the product kernel


// One rank panel (at most PROD_RANK rank rows) of a long low-rank block by the CTA, complex64:
// the warps take 64 columns of a panel side each in turn, the intermediates are summed over the
// warps in shared memory, and the second reading of the panel hits L1.  One warp for the panel
// is a serial chain of (m + n) / 16 loads, 8 in flight (30,720-unknown sphere, level 2, 219
// panels: 50 us, one warp each, 16 us).
__device__ __noinline__ void lowrank_panel(const Item &it, const float2 *__restrict__ pool,
                                              const float2 *__restrict__ x, float2 *__restrict__ z,
                                              float2 (*ts)[2 * PROD_RANK], int lane, int w)
{
    static_assert(PROD_RANK == 8, "reduce8");
    const int k = it.k;
    const float2 *F[2] = {pool + it.off, pool + it.off + panel_voff(it)};
    const int len[2] = {it.m, it.n}, at[2] = {it.row0, it.col0};
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        float2 t[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) t[l] = make_float2(0.f, 0.f);
        for (int i = 64 * w + 2 * lane; i < len[side]; i += 64 * APPLY_WARPS) {
            const Pair<float> p = ld_vec(x + at[side] + i);
#pragma unroll
            for (int l = 0; l < 8; ++l)
                if (l < k) {
                    const Pair<float> a = ld_cached(F[side] + (int64_t)l * len[side] + i);
                    cfma(t[l], a.a, p.a);
                    cfma(t[l], a.b, p.b);
                }
        }
        reduce8<float2>(t, lane);
        if (lane < 8) ts[w][8 * side + lane] = t[0];
    }
    __syncthreads();
    // lane 8 side + l: the intermediate of rank row l (0: U^T x_I, 1: V x_J)
    float2 tot = make_float2(0.f, 0.f);
    if (lane < 16)
        for (int q = 0; q < APPLY_WARPS; ++q) tot = cadd(tot, ts[q][lane]);
#pragma unroll
    for (int side = 0; side < 2; ++side) {
        float2 f[8];
#pragma unroll
        for (int l = 0; l < 8; ++l) f[l] = shfl_idx(tot, 8 * (1 - side) + l);
        for (int i = 64 * w + 2 * lane; i < len[side]; i += 64 * APPLY_WARPS) {
            float2 o0 = make_float2(0.f, 0.f), o1 = o0;
#pragma unroll
            for (int l = 0; l < 8; ++l)
                if (l < k) {
                    const Pair<float> a = ld_cached(F[side] + (int64_t)l * len[side] + i);
                    cfma(o0, a.a, f[l]);
                    cfma(o1, a.b, f[l]);
                }
            red2(z + at[side] + i, o0, o1);
        }
    }
}

// MINB: CTAs per SM the register budget must allow (3 for complex64, so that 24
// warps per SM stream blocks; 1 for the FP64 comparator path, which needs more
// registers)
// LONG: the warps' items may be longer than 64
template <class T, class A, int MINB, bool LONG>
__global__ void __launch_bounds__(APPLY_WARPS * 32, MINB)
k_apply_items(const Item *__restrict__ items, int64_t n_items, const Item *__restrict__ panels, int wide, const typename CT<T>::C *__restrict__ pool,
              const typename CT<T>::C *__restrict__ x, int64_t ldx, typename CT<A>::C *__restrict__ z,
              int64_t ldz, int nrhs)
{
    using CTy = typename CT<T>::C;
    __shared__ CTy xs_all[APPLY_WARPS][32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    if constexpr (sizeof(T) == 4) {
        // the first `wide` CTAs: one panel of a long low-rank block and one right-hand side each
        __shared__ float2 ts[APPLY_WARPS][2 * PROD_RANK];
        if ((int)blockIdx.x < wide) {
            const int r = blockIdx.x % nrhs;
            lowrank_panel(panels[blockIdx.x / nrhs], pool, x + r * ldx, z + r * ldz, ts, lane, w);
            return;
        }
    }
    const int nw = ((int)gridDim.x - wide) * APPLY_WARPS;
    for (int64_t t = (int64_t)((int)blockIdx.x - wide) * APPLY_WARPS + w; t < n_items; t += nw) {
        const Item it = items[t];
        for (int r = 0; r < nrhs; ++r) {
            if (it.k == 0)
                dense_item<T, A>(it, pool, x + r * ldx, z + r * ldz, xs_all[w], lane);
            else
                lowrank_item<T, A, LONG>(it, LONG && sizeof(T) == 4 ? panel_voff(it) : (int64_t)it.k * it.m, pool,
                                         x + r * ldx, z + r * ldz, lane);
        }
    }
}

template <class T, class A, int MINB>
int apply_grid(hm_matrix h)
{
    static int per_sm = -1;
    if (per_sm < 0) {
        int v = 0;
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&v, k_apply_items<T, A, MINB, true>, APPLY_WARPS * 32, 0);
        per_sm = v > 0 ? v : 1;
    }
    return per_sm * (h->num_sms > 0 ? h->num_sms : 1);
}

} // namespace

int64_t product_warps(hm_matrix h)
{
    if (h->num_sms <= 0) {
        int dev = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&h->num_sms, cudaDevAttrMultiProcessorCount, dev);
    }
    return (int64_t)apply_grid<float, float, 3>(h) * APPLY_WARPS;
}

int launch_apply_items(hm_matrix h, const LevelList &L, const void *x, void *z, int nrhs, bool fp64,
                       cudaStream_t s, int rb)
{
    const int64_t n = (int64_t)L.items.size();
    if (n == 0) return 0;
    if (fp64) {
        int g = apply_grid<double, double, 1>(h);
        if ((int64_t)g * APPLY_WARPS > n) g = (int)((n + APPLY_WARPS - 1) / APPLY_WARPS);
        k_apply_items<double, double, 1, true><<<g, APPLY_WARPS * 32, 0, s>>>(
            L.d_items, n, nullptr, 0, h->d_pool64, (const double2 *)x, h->pN, (double2 *)z, h->pN, nrhs);
        return 1;
    } else {
        int launched = 0;
        // tall dense blocks go as row panels, long low-rank ones as rank panels (LevelList::d_prod), one warp each
        const Item *list = L.d_prod;
        int64_t cnt = L.n_prod - L.n_prod_wide;
        if (rb < 0) rb = nrhs < MRHS_MIN_RHS ? 0 : nrhs <= 8 ? 8 : 16;
        if (rb == RB_TC && nrhs > 1) {
            // the small blocks (dense and low-rank) on the tensor cores
            launched += launch_apply_tc(h, L, (const float2 *)x, (float2 *)z, nrhs, s);
            list = L.d_prod_big;
            cnt = L.n_prod_big - L.n_prod_wide;
            if (L.n_prod_big == 0) return launched;
        } else if (rb > 0 && nrhs > 1 && L.n_small > 0) {
            // many right-hand sides: on the matrix instructions, or blocks staged in shared memory once per chunk
            if (rb == 32 && L.mm_built && h->ws.d_mm && h->ws.mm_bytes >= mm_ws_bytes(L, nrhs, false)) {
                launched += launch_mm_product(h, L, (const float2 *)x, (float2 *)z, nrhs, h->ws.d_mm, s);
            } else {
                launch_apply_items_mrhs(h, L, (const float2 *)x, (float2 *)z, nrhs, std::min(rb, 16), s);
                launched += 1;
            }
            list = L.d_prod_big;
            cnt = L.n_prod_big - L.n_prod_wide;
            if (L.n_prod_big == 0) return launched;
        }
        const int64_t wide = L.n_prod_wide * nrhs;
        const int64_t g = std::min<int64_t>(apply_grid<float, float, 3>(h), (cnt + APPLY_WARPS - 1) / APPLY_WARPS);
        const auto kern = L.prod_long ? k_apply_items<float, float, 3, true> : k_apply_items<float, float, 3, false>;
        kern<<<(unsigned)(wide + g), APPLY_WARPS * 32, 0, s>>>(
            list + L.n_prod_wide, cnt, list, (int)wide, h->d_pool32, (const float2 *)x, h->pN, (float2 *)z, h->pN, nrhs);
        return launched + 1;
    }
}

} // namespace hm
