// FP64-class residual products for many right-hand sides, owner-computes form
// (the refinement residual r = b - A_m x of the solve; the block products are
// eq. 6 and eq. 8 of arxiv 2307.03968 with the half storage of §III).
//
// A work unit is one output cluster O of a level, or a part of its products where there are few
// clusters (split_owner_units: 7,500 unknowns, 128 clusters, 50 right-hand sides: 512 whole units
// leave the 608 places of the chip a single uneven wave), and one group of RG right-hand
// sides (16, or 8 for calls with few right-hand sides).  The CTA walks the directed products into O (the stored
// blocks with O as row cluster, and mirrored, those with O as column cluster;
// dense or low-rank), in a fixed order, and keeps the sums in registers as
// double-float complex numbers.  Each directed product is summed, per output row
// and right-hand side, as one error-free chain on a common grid (k_dot2.cuh: every
// product rounded exactly onto a power-of-two grid whose sigma comes from the
// product's precomputed bound, k_prod_bounds, and the input's largest component;
// the remainders summed apart), folded once into the double-float sum with a
// compensated addition.  Thread t of the RT-thread CTA (RT = 128 or 256) owns
// output row t % 64 and the right-hand sides QN (t / 64) .. + QN - 1 of the group,
// QN = RG / (RT / 64).  The unit's sums are stored once, in FP64, into the level's
// [RHS][pN] array: no partial slots, no atomics, and the result is independent of
// scheduling.  k_gather_own then forms b - (D x + sum over levels) in FP64.
//
// Shared-memory staging keeps every compute read consecutive along the output
// row: a dense block is stored K-major (element (K index j, output i) at
// j * 65 + i), whichever orientation the product reads it in; a low-rank
// block's input-side factor W is stored K-major over its rank rows and its
// output-side factor Y rank-major.
#include "k_dot2.cuh"

#include <algorithm>

namespace hm {
namespace {

using namespace kc;
using namespace dot2;
constexpr int RGMAX = 16;        // right-hand sides per unit (at most)
constexpr int BS = 65;           // float2 stride of a staged K row of a block (odd: conflict-free staging)
constexpr int WS = 33;           // float2 stride of a staged K row of W (rank <= 32)
constexpr int XP = 9;            // float4 stride of a staged K row of x (8 pairs of right-hand sides)
constexpr int SM_B = 64 * WS + 32 * BS;   // float2: W (64 x WS) then Y (32 x BS), or a dense block (64 x BS)
constexpr int SM_X = 64 * XP;
constexpr int SM_T = 32 * RGMAX; // float4: T = W x (rank x RG / 2 pairs of RHS x leading and trailing parts)
static_assert(64 * BS <= SM_B, "a dense block fits the block area");

struct alignas(16) Smem {
    float2 b[SM_B];
    float4 x[SM_X];
    float4 t[SM_T];
    float mx[2 * RGMAX];         // max |x|_inf over K indices 32h..32h+31 (h = 0, 1), per right-hand side
};

// The chains of two right-hand sides q, q + 1 as packed pairs (k_dot2.cuh xstep): x is staged as
// (re_q, re_q+1, im_q, im_q+1), so that the right-hand sides need no rearranged copies, and the
// block element's duplicated parts serve all of a thread's pairs.  8 instructions a complex
// product and right-hand side instead of 16: 0.845 to 0.677 ms (with the parts) at 7,500 unknowns, 50 right-hand sides.
struct chain2 { float2 tr, rr, ti, ri; };   // real part: grid sum, remainder; imaginary part
__device__ __forceinline__ void c2_start(chain2 &c, float2 sigma) { c = {sigma, dup(0.f), sigma, dup(0.f)}; }
__device__ __forceinline__ void step2(float2 &tau, float2 &r, float2 a, float2 b)
{
    const float2 t2 = fma2(a, b, tau);
    r = add2(r, fma2(a, b, sub2(tau, t2)));
    tau = t2;
}
// c += a x for a block element a and the pair's x
__device__ __forceinline__ void c2_step(chain2 &c, float2 a, float4 x)
{
    const float2 re = make_float2(x.x, x.y), im = make_float2(x.z, x.w);
    step2(c.tr, c.rr, dup(a.x), re);
    step2(c.tr, c.rr, dup(-a.y), im);
    step2(c.ti, c.ri, dup(a.x), im);
    step2(c.ti, c.ri, dup(a.y), re);
}
// the trailing parts of a double-float x into the remainders
__device__ __forceinline__ void c2_lo(chain2 &c, float2 a, float4 x)
{
    const float2 re = make_float2(x.x, x.y), im = make_float2(x.z, x.w);
    c.rr = fma2(dup(-a.y), im, fma2(dup(a.x), re, c.rr));
    c.ri = fma2(dup(a.y), re, fma2(dup(a.x), im, c.ri));
}
__device__ __forceinline__ void c2_fold(cdf (&acc)[2], const chain2 &c, float2 sigma)
{
    const float2 gr = sub2(c.tr, sigma), gi = sub2(c.ti, sigma);
    acc[0] = cdf_add(acc[0], {{gr.x, c.rr.x}, {gi.x, c.ri.x}});
    acc[1] = cdf_add(acc[1], {{gr.y, c.rr.y}, {gi.y, c.ri.y}});
}

// stage x of the input cluster: pair q / 2 of xs[j * XP + ..] = x[(r0 + q) * ldx + in0 + j] for j < klen, q < nr,
// 0 for the rest of j < roundup4(klen); mx[2 q + h] = max over j = 32h..32h+31 of |x|_inf.
// Every thread runs the same number of iterations (RG * 64 is a multiple of RT), and a warp
// covers 32 consecutive j of one q.
template <int RG, int RT>
__device__ __forceinline__ void stage_x(float4 *xs, float *mx, const float2 *__restrict__ x, int64_t ldx, int r0,
                                        int nr, int in0, int klen)
{
    static_assert((RG * 64) % RT == 0, "uniform staging loop");
    const int k4 = (klen + 3) & ~3;
    for (int e = threadIdx.x; e < RG * 64; e += RT) {
        const int q = e >> 6, j = e & 63;
        const float2 v = (j < klen && q < nr) ? x[(int64_t)(r0 + q) * ldx + in0 + j] : make_float2(0.f, 0.f);
        if (j < k4) {
            float *d = reinterpret_cast<float *>(xs + j * XP + (q >> 1)) + (q & 1);
            d[0] = v.x;
            d[2] = v.y;
        }
        const float m = warp_max(linf(v));
        if ((j & 31) == 0) mx[2 * q + (j >> 5)] = m;
    }
}
// the largest |x|_inf of right-hand side q over the staged input
__device__ __forceinline__ float x_max(const float *mx, int q) { return fmaxf(mx[2 * q], mx[2 * q + 1]); }

template <int RG, int RT>
__global__ void __launch_bounds__(RT, 4)
k_resid_own(const RcUnit *__restrict__ units, int n_units, const TcProd *__restrict__ prods,
            const float2 *__restrict__ pbnd, const float2 *__restrict__ pool, const float2 *__restrict__ x,
            int64_t ldx, int nrhs, double2 *__restrict__ own, int64_t ldo, int64_t lstride)
{
    extern __shared__ __align__(16) unsigned char smraw[];
    Smem &S = *reinterpret_cast<Smem *>(smraw);
    constexpr int QN = RG / (RT / 64);   // right-hand sides per thread
    const int tid = threadIdx.x, i = tid & 63, hh = tid >> 6;
    const int n_groups = (nrhs + RG - 1) / RG;
    const int64_t total = (int64_t)n_units * n_groups;
    // cluster-major: the RHS groups of one output cluster are consecutive units, so they
    // run on neighbouring CTAs at the same time and read the cluster's blocks from DRAM
    // once between them (the later reads hit L2)
    for (int64_t u = blockIdx.x; u < total; u += gridDim.x) {
        const RcUnit U = units[u / n_groups];
        const int r0 = (int)(u % n_groups) * RG, nr = min(RG, nrhs - r0);
        cdf acc[QN / 2][2];
#pragma unroll
        for (int q = 0; q < QN; ++q) acc[q / 2][q & 1] = cdf_zero();
        for (int p = U.p0; p < U.p1; ++p) {
            const TcProd P = prods[p];
            __syncthreads();                                  // the previous product's reads are done
            stage_x<RG, RT>(S.x, S.mx, x, ldx, r0, nr, P.in0, P.klen);
            if (P.rank == 0) {
                // block elements (output i < olen, K j < klen) into b[j * BS + i]
                const float2 *B = pool + P.b_off;
                const int rows = P.trans ? P.klen : P.olen;
                for (int e = tid; e < rows * 64; e += RT) {
                    const int a = e >> 6, c = e & 63;         // source row a, column c (coalesced along c)
                    if (P.trans) {                            // element (i = c, j = a) = B[a][c]
                        if (a < P.klen && c < P.olen) S.b[a * BS + c] = B[(int64_t)a * P.b_ld + c];
                    } else {                                  // element (i = a, j = c) = B[a][c]
                        if (a < P.olen && c < P.klen) S.b[c * BS + a] = B[(int64_t)a * P.b_ld + c];
                    }
                }
                __syncthreads();
                if (i < P.olen) {
                    // one chain per right-hand side over all K indices, on the grid of the
                    // product's largest output-row 1-norm times the input's largest component
                    const float bo = pbnd[p].x;
                    float2 sg[QN / 2];
                    chain2 c[QN / 2];
#pragma unroll
                    for (int q = 0; q < QN / 2; ++q) {
                        sg[q] = make_float2(grid_sigma(bo, x_max(S.mx, QN * hh + 2 * q)),
                                            grid_sigma(bo, x_max(S.mx, QN * hh + 2 * q + 1)));
                        c2_start(c[q], sg[q]);
                    }
                    const float4 *xv = S.x + QN / 2 * hh;
#pragma unroll 4
                    for (int j = 0; j < P.klen; ++j) {
                        const float2 bv = S.b[j * BS + i];
#pragma unroll
                        for (int q = 0; q < QN / 2; ++q) c2_step(c[q], bv, xv[j * XP + q]);
                    }
#pragma unroll
                    for (int q = 0; q < QN / 2; ++q) c2_fold(acc[q], c[q], sg[q]);
                }
            } else {
                // W (rank rows l, K j) into b[j * WS + l]; Y (element (i, l) = Y[l][i]) into y[l * BS + i]
                float2 *Wsm = S.b, *Ysm = S.b + 64 * WS;
                const float2 *W = pool + P.b_off, *Y = pool + P.y_off;
                for (int e = tid; e < P.rank * 64; e += RT) {
                    const int l = e >> 6, c = e & 63;
                    if (c < P.klen) Wsm[c * WS + l] = W[(int64_t)l * P.b_ld + c];
                    if (c < P.olen) Ysm[l * BS + c] = Y[(int64_t)l * P.y_ld + c];
                }
                __syncthreads();
                // stage 1: T[l][q] = sum_j W[l][j] x[j][q]; thread (row l0 + lr, pair qp, K slice
                // ks: j = ks, ks + NS, ...); the slices' chains share the grid of W's largest rank-row
                // 1-norm times x's largest component, so their grid parts add exactly across lanes
                const float2 bb = pbnd[p];
                {
                    constexpr int NS = RG == 16 ? 2 : 4;           // K slices per rank row and pair
                    constexpr int LR = RT / (NS * RG / 2);         // rank rows per round
                    const int ks = tid % NS, qp = (tid / NS) % (RG / 2), lr = tid / (NS * RG / 2);
                    const float2 s1 = make_float2(grid_sigma(bb.x, x_max(S.mx, 2 * qp)),
                                                  grid_sigma(bb.x, x_max(S.mx, 2 * qp + 1)));
                    for (int l0 = 0; l0 < P.rank; l0 += LR) {
                        const int l = l0 + lr;
                        chain2 c;
                        c2_start(c, s1);
                        if (l < P.rank)
                            for (int j = ks; j < P.klen; j += NS) c2_step(c, Wsm[j * WS + l], S.x[j * XP + qp]);
                        const float2 gr = sub2(c.tr, s1), gi = sub2(c.ti, s1);
                        float v[8] = {gr.x, gr.y, gi.x, gi.y, c.rr.x, c.rr.y, c.ri.x, c.ri.y};
#pragma unroll
                        for (int sh = 1; sh < NS; sh <<= 1)
#pragma unroll
                            for (int e = 0; e < 8; ++e) v[e] = __fadd_rn(v[e], __shfl_xor_sync(FULL, v[e], sh));
                        if (ks == 0 && l < P.rank) {
                            S.t[l * RG + 2 * qp] = make_float4(v[0], v[1], v[2], v[3]);
                            S.t[l * RG + 2 * qp + 1] = make_float4(v[4], v[5], v[6], v[7]);
                        }
                    }
                }
                __syncthreads();
                // stage 2: out[i][q] += sum_l Y[i][l] T[l][q], one chain per right-hand side over
                // all rank rows: the leading part of T[l][q] is a grid sum, at most half of
                // stage 1's sigma, which bounds the inputs with Y's largest output-row 1-norm
                if (i < P.olen) {
                    float2 sg[QN / 2];
                    chain2 c[QN / 2];
#pragma unroll
                    for (int q = 0; q < QN / 2; ++q) {
                        const int g = QN * hh + 2 * q;
                        sg[q] = make_float2(grid_sigma(bb.y, 0.5f * grid_sigma(bb.x, x_max(S.mx, g))),
                                            grid_sigma(bb.y, 0.5f * grid_sigma(bb.x, x_max(S.mx, g + 1))));
                        c2_start(c[q], sg[q]);
                    }
                    for (int l = 0; l < P.rank; ++l) {
                        const float2 yv = Ysm[l * BS + i];
#pragma unroll
                        for (int q = 0; q < QN / 2; ++q) {
                            const float4 *t = S.t + l * RG + QN * hh + 2 * q;
                            c2_step(c[q], yv, t[0]);
                            c2_lo(c[q], yv, t[1]);
                        }
                    }
#pragma unroll
                    for (int q = 0; q < QN / 2; ++q) c2_fold(acc[q], c[q], sg[q]);
                }
            }
        }
        if (i < U.mlen) {
#pragma unroll
            for (int q = 0; q < QN; ++q) {
                const int r = QN * hh + q;
                if (r < nr) own[U.part * lstride + (int64_t)(r0 + r) * ldo + U.out0 + i] = to_d2(acc[q / 2][q & 1]);
            }
        }
    }
}

// Dot2 of two right-hand sides as packed pairs (k_dot2.cuh dot2): acc += a * b, na = -a
struct dot2x2 { float2 hi, lo; };
__device__ __forceinline__ void dot2_pair(dot2x2 &acc, float2 a, float2 na, float2 b)
{
    const float2 z = dup(0.f);
    const float2 p = fma2(a, b, z), np = fma2(na, b, z);
    const float2 s = add2(acc.hi, p), bb = sub2(s, acc.hi);
    const float2 q = add2(sub2(acc.hi, sub2(s, bb)), sub2(p, bb));
    acc.lo = add2(acc.lo, add2(q, fma2(a, b, np)));
    acc.hi = s;
}

// Per leaf (blockIdx.x) and GR right-hand sides (blockIdx.y): acc = D_I x_I (Dot2) +
// the `arrays` owner sums at the leaf's rows (FP64), in a fixed order.  If b
// is given, out = b - acc (FP64, rounded to complex64) and |r|^2, |b|^2 go to
// norms; else out = acc (complex64).  x of the leaf is staged in dynamic shared
// memory as pairs; each element of D_I serves the GR right-hand sides.  Four threads share a
// row: columns j = js, js + 4, .. each, then right-hand side q = js each (the Dot2 chain over
// the columns is what a row waits for).  7,500 unknowns, 50 right-hand sides: 54 us with one a
// CTA and a thread a row, 29 us.
template <int GR>
__global__ void __launch_bounds__(256)
k_gather_own(const int32_t *__restrict__ pleaf_off, const int64_t *__restrict__ dinv_off,
             const float2 *__restrict__ self32, const float2 *__restrict__ x, int64_t ld, int nrhs, int arrays,
             const double2 *__restrict__ own, int64_t lstride, const float2 *__restrict__ b, float2 *__restrict__ out,
             double *norms)
{
    static_assert(GR == 1 || GR == 4, "a right-hand side per column slice");
    constexpr int GP = (GR + 1) / 2;
    __shared__ cdf part[4][GR][64];
    extern __shared__ __align__(16) unsigned char gsm[];
    float *xs = reinterpret_cast<float *>(gsm);
    const int leaf = blockIdx.x, r0 = GR * blockIdx.y, tid = threadIdx.x, lane = tid & 31, js = tid >> 6;
    const int o = pleaf_off[leaf], np = pleaf_off[leaf + 1] - o;
    const int r = r0 + js;                                     // the thread's right-hand side
    const bool mine = js < GR && r < nrhs;
    for (int e = tid; e < 2 * GP * np; e += 256) {
        const int q = e / np, j = e - q * np;
        const float2 v = q < GR && r0 + q < nrhs ? x[(r0 + q) * ld + o + j] : make_float2(0.f, 0.f);
        float *d = xs + 4 * (j * GP + (q >> 1)) + (q & 1);
        d[0] = v.x;
        d[2] = v.y;
    }
    __syncthreads();
    const float4 *xp = reinterpret_cast<const float4 *>(xs);
    const float2 *Sd = self32 + dinv_off[leaf];                 // column-major np x np
    double rr = 0.0, bb = 0.0;
    for (int i0 = 0; i0 < np; i0 += 64) {
        const int i = i0 + (tid & 63);
        if (i < np) {
            dot2x2 re[GP], im[GP];
#pragma unroll
            for (int q = 0; q < GP; ++q) re[q] = im[q] = {dup(0.f), dup(0.f)};
#pragma unroll 4
            for (int j = js; j < np; j += 4) {
                const float2 a = Sd[(int64_t)j * np + i];
#pragma unroll
                for (int q = 0; q < GP; ++q) {
                    const float4 v = xp[j * GP + q];
                    const float2 vr = make_float2(v.x, v.y), vi = make_float2(v.z, v.w);
                    dot2_pair(re[q], dup(a.x), dup(-a.x), vr);
                    dot2_pair(re[q], dup(-a.y), dup(a.y), vi);
                    dot2_pair(im[q], dup(a.x), dup(-a.x), vi);
                    dot2_pair(im[q], dup(a.y), dup(-a.y), vr);
                }
            }
#pragma unroll
            for (int q = 0; q < GR; ++q) {
                const dot2x2 &u = re[q / 2], &v = im[q / 2];
                part[js][q][tid & 63] =
                    q & 1 ? cdf{{u.hi.y, u.lo.y}, {v.hi.y, v.lo.y}} : cdf{{u.hi.x, u.lo.x}, {v.hi.x, v.lo.x}};
            }
        }
        __syncthreads();
        if (i < np && mine) {
            const int64_t g = r * ld + o + i;
            cdf s = part[0][js][tid & 63];
#pragma unroll
            for (int q = 1; q < 4; ++q) s = cdf_add(s, part[q][js][tid & 63]);
            double2 acc = to_d2(s);
            for (int lev = 0; lev < arrays; ++lev) acc = cadd(acc, own[lev * lstride + g]);
            if (b) {
                const double2 bv = conv<double2>(b[g]);
                const double2 rv = csub(bv, acc);
                out[g] = make_float2((float)rv.x, (float)rv.y);
                rr += rv.x * rv.x + rv.y * rv.y;
                bb += bv.x * bv.x + bv.y * bv.y;
            } else {
                out[g] = make_float2((float)acc.x, (float)acc.y);
            }
        }
        __syncthreads();
    }
    if (norms && mine) {                                       // whole warps: js is a warp's
        for (int s = 16; s >= 1; s >>= 1) {
            rr += __shfl_xor_sync(FULL, rr, s);
            bb += __shfl_xor_sync(FULL, bb, s);
        }
        if (lane == 0) {
            atomicAdd(&norms[2 * r], rr);
            atomicAdd(&norms[2 * r + 1], bb);
        }
    }
}

// Per directed product, the bounds its common grids take (k_resid_own): x = the
// largest 1-norm of an output row of the oriented block (dense) or of a rank row of
// the input-side factor W (low-rank, stage 1); y = the largest 1-norm, over the rank
// rows, of an output row of Y (low-rank, stage 2).  FP64 sums rounded up; one warp
// per product.
__global__ void __launch_bounds__(256)
k_prod_bounds(const TcProd *__restrict__ prods, int64_t n, const float2 *__restrict__ pool, float2 *__restrict__ out)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t t = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); t < n; t += nw) {
        const TcProd P = prods[t];
        double a = 0.0, b = 0.0, c = 0.0, d = 0.0;
        if (P.rank == 0) {
            if (P.trans) l1_bounds(pool + P.b_off, P.klen, P.olen, P.b_ld, c, a, lane);   // output i = column i
            else l1_bounds(pool + P.b_off, P.olen, P.klen, P.b_ld, a, c, lane);
        } else {
            l1_bounds(pool + P.b_off, P.rank, P.klen, P.b_ld, a, c, lane);
            l1_bounds(pool + P.y_off, P.rank, P.olen, P.y_ld, d, b, lane);
        }
        if (lane == 0) out[t] = make_float2(__double2float_ru(a), __double2float_ru(b));
    }
}

} // namespace

void launch_prod_bounds(const TcProd *prods, int64_t n, const float2 *pool, float2 *out, cudaStream_t s)
{
    if (n <= 0) return;
    const int g = (int)std::min<int64_t>((n + 7) / 8, 152 * 16);
    k_prod_bounds<<<g, 256, 0, s>>>(prods, n, pool, out);
}

// owner-computes FP64-class products of a level's small items: the sum over the level's parts q of
// own[q * lstride + r * pN + i] = (M_level x_r)_i for the level's output rows (a level whose items
// are all small; the rest of own is untouched)
void launch_resid_own(hm_matrix h, const LevelList &L, const float2 *x, double2 *own, int64_t lstride, int nrhs,
                      cudaStream_t s)
{
    if (L.n_rcu == 0 || nrhs <= 0) return;
    constexpr int SMEM = (int)sizeof(Smem);
    static bool attr = false;
    if (!attr) {
        for (const void *f : {(const void *)k_resid_own<8, 128>, (const void *)k_resid_own<16, 128>,
                              (const void *)k_resid_own<8, 256>, (const void *)k_resid_own<16, 256>}) {
            cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, SMEM);
            cudaFuncSetAttribute(f, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        }
        attr = true;
    }
    // groups of 8 right-hand sides up to 32 of them, so that small calls still have enough units.
    // four CTAs of ~50 KB per SM: of 256 threads (4 RHS per thread, 64 registers) up to 128 RHS,
    // of 128 threads (8 RHS per thread) above: measured on the 30,720-unknown sphere, 0.499 /
    // 0.365 ms per RHS at 16 / 64 RHS against 0.587 / 0.406 for 128 threads, and 0.382 against
    // 0.386 for 256 threads at 181
    const int rg = nrhs <= 32 ? 8 : 16;
    const bool wide = nrhs <= 128;
    const int64_t units = L.n_rcu * (int64_t)((nrhs + rg - 1) / rg);
    int64_t g = 4 * (int64_t)(h->num_sms > 0 ? h->num_sms : 1);
    if (g > units) g = units;
    auto go = [&](auto kern, int rt) {
        kern<<<(unsigned)g, rt, SMEM, s>>>(L.d_rcu, (int)L.n_rcu, L.d_rcp, L.d_rcb, h->d_pool32, x, h->pN, nrhs, own,
                                           h->pN, lstride);
    };
    if (rg == 8) wide ? go(k_resid_own<8, 256>, 256) : go(k_resid_own<8, 128>, 128);
    else wide ? go(k_resid_own<16, 256>, 256) : go(k_resid_own<16, 128>, 128);
}

void launch_gather_own(hm_matrix h, const float2 *x, int arrays, const double2 *own, int64_t lstride, const float2 *b,
                       float2 *out, double *norms, int nrhs, cudaStream_t s)
{
    int64_t maxnp = 0;
    for (int64_t i = 0; i < h->n_leaves; ++i) maxnp = std::max<int64_t>(maxnp, h->pleaf_off[i + 1] - h->pleaf_off[i]);
    // four right-hand sides a CTA where that leaves a CTA per SM
    const int64_t groups = (nrhs + 3) / 4;
    const bool four = h->n_leaves * groups >= h->num_sms;
    const auto kern = four ? k_gather_own<4> : k_gather_own<1>;
    const size_t sm = sizeof(float4) * (four ? 2 : 1) * (size_t)std::max<int64_t>(maxnp, 1);
    // the attribute is of the current device, so it is set by every call that needs it (leaves of more
    // than 1,024 unknowns; the longest, 1,536, take 48 KB beside the 16 KB of sums)
    if (sm > 32 * 1024) cudaFuncSetAttribute(k_gather_own<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    kern<<<dim3((unsigned)h->n_leaves, (unsigned)(four ? groups : nrhs)), 256, sm, s>>>(
        h->d_pleaf_off, h->d_dinv_off, h->d_self32, x, h->pN, nrhs, arrays, own, lstride, b, out, norms);
}

} // namespace hm
