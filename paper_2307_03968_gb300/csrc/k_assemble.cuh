// Basis-independent parts of the GPU H-Matrix construction (arxiv 2307.03968
// §III, eqs. 6-7), shared by the surface (RWG) and volume (SWG) builds.
//
//   k_fill       near-field blocks (complex64) and leaf self blocks
//                (complex128, upper half filled and mirrored) from the basis
//                geometry's entry function;
//   k_aca        partially pivoted adaptive cross approximation of every far
//                block, one CTA per block (§III, refs. [22,23]);
//   k_recompress re-compression of each ACA pair (ref. [24]): QR of both
//                factors by twice-iterated Gram-Schmidt, SVD of the small core
//                by one-sided Jacobi rotations, truncation at the tolerance;
//   k_pack_far   copy of the compressed factors into the padded pool;
//   host         cluster tree, eq. 7 block partition and the packed layout.
//
// A basis geometry G is a struct of device pointers with a member `perm`
// (tree position -> original unknown) and a device member template
//   template <class R> CX<R> entry(int m, int n) const
// returning the Galerkin matrix entry Z[m][n] of original unknowns m, n.
#pragma once

#include "hm_internal.h"

#include <algorithm>
#include <array>
#include <cmath>
#include <cstring>
#include <numeric>

namespace hm {
namespace {

constexpr int ACA_THREADS = 128;
constexpr int ACA_KCAP = 48;
constexpr int RC_THREADS = 256;

template <class R> struct CX { R re, im; };

// entry Z[m][n] in FP32 by G::PARTS neighbouring lanes, lane `part` evaluating its part; the
// parts are added in the order of entry(), to the same result, in every lane (all lanes of
// the warp take part)
template <class G> __device__ __forceinline__ CX<float> entry_parts(const G &g, int m, int n, int part)
{
    if constexpr (G::PARTS == 1) {
        return g.template entry<float>(m, n);
    } else {
        const CX<float> v = g.part(m, n, part);
        CX<float> z{0, 0};
        const int base = (threadIdx.x & 31) - part;
#pragma unroll
        for (int p = 0; p < G::PARTS; ++p) {
            z.re += __shfl_sync(0xffffffffu, v.re, base + p);
            z.im += __shfl_sync(0xffffffffu, v.im, base + p);
        }
        return g.scale(m, n, z);
    }
}

__device__ __forceinline__ float sqrtR(float v) { return sqrtf(v); }
__device__ __forceinline__ double sqrtR(double v) { return sqrt(v); }
__device__ __forceinline__ float logR(float v) { return logf(v); }
__device__ __forceinline__ double logR(double v) { return log(v); }
__device__ __forceinline__ float atanR(float v) { return atanf(v); }
__device__ __forceinline__ double atanR(double v) { return atan(v); }
__device__ __forceinline__ void sincosR(float v, float *s, float *c) { sincosf(v, s, c); }
__device__ __forceinline__ void sincosR(double v, double *s, double *c) { sincos(v, s, c); }
__device__ __forceinline__ float sinR(float v) { return sinf(v); }
__device__ __forceinline__ double sinR(double v) { return sin(v); }
__device__ __forceinline__ float absR(float v) { return fabsf(v); }
__device__ __forceinline__ double absR(double v) { return fabs(v); }

// ---------------------------------------------------------------- fill ----------
struct FillJob {
    int64_t out;     // element offset (pool for near, self64 for self)
    int64_t first;   // first flat entry index of this job
    int32_t r0, c0;  // tree positions of the row / column leaf starts
    int32_t m, n;    // true sizes
    int32_t ld;      // output row stride (near) ; unused for self
    int32_t self;    // 1 = self block (complex128, upper half + mirror)
};

// One thread per entry.  SELF = false: complex64 near blocks (row-major, row
// stride ld); SELF = true: complex128 leaf self blocks, the upper triangle
// (i <= j) enumerated row by row and mirrored.  Separate instantiations keep
// the FP32 near fill free of the FP64 path's registers.
template <class G, bool SELF>
__global__ void k_fill(G g, const FillJob *__restrict__ jobs, int njobs, int64_t total, float2 *pool,
                       double2 *self64)
{
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < total;
         t += (int64_t)gridDim.x * blockDim.x) {
        int lo = 0, hi = njobs - 1;
        while (lo < hi) {   // last job with first <= t
            const int mid = (lo + hi + 1) >> 1;
            if (jobs[mid].first <= t) lo = mid; else hi = mid - 1;
        }
        const FillJob J = jobs[lo];
        const int64_t e = t - J.first;
        if (SELF) {
            int i = 0;
            int64_t rem = e;
            while (rem >= J.n - i) { rem -= J.n - i; ++i; }
            const int j = i + (int)rem;
            const CX<double> v = g.template entry<double>(g.perm[J.r0 + i], g.perm[J.c0 + j]);
            self64[J.out + (int64_t)i * J.n + j] = make_double2(v.re, v.im);
            if (i != j) self64[J.out + (int64_t)j * J.n + i] = make_double2(v.re, v.im);
        } else {
            const int i = (int)(e / J.n), j = (int)(e - (int64_t)i * J.n);
            const CX<float> v = g.template entry<float>(g.perm[J.r0 + i], g.perm[J.c0 + j]);
            pool[J.out + (int64_t)i * J.ld + j] = make_float2(v.re, v.im);
        }
    }
}

// ---------------------------------------------------------------- ACA -----------
struct AcaJob {
    int64_t off;     // scratch offset: U^T (kmax x m) then V (kmax x n)
    int32_t r0, c0;  // tree positions
    int32_t m, n, kmax, pad;
};

__device__ __forceinline__ float cabs2(float2 a) { return a.x * a.x + a.y * a.y; }
__device__ __forceinline__ float2 cmulf(float2 a, float2 b) { return make_float2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ float2 cconjmul(float2 a, float2 b)   // conj(a) * b
{
    return make_float2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x);
}

// block-wide argmax of v (ties: lowest index); returns (value, index) to all threads
__device__ void block_argmax(float v, int idx, float *sv, int *si, float &ov, int &oi)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = blockDim.x >> 5;
    for (int s = 16; s >= 1; s >>= 1) {
        const float v2 = __shfl_xor_sync(0xffffffffu, v, s);
        const int i2 = __shfl_xor_sync(0xffffffffu, idx, s);
        if (v2 > v || (v2 == v && i2 < idx)) { v = v2; idx = i2; }
    }
    __syncthreads();
    if (lane == 0) { sv[w] = v; si[w] = idx; }
    __syncthreads();
    ov = sv[0];
    oi = si[0];
    for (int q = 1; q < nw; ++q)
        if (sv[q] > ov || (sv[q] == ov && si[q] < oi)) { ov = sv[q]; oi = si[q]; }
}

// warp-wide sums (FP64 accumulation of FP32 products) over conj(a[i]) b[i], i < n
__device__ __forceinline__ double2 warp_cdot(const float2 *a, const float2 *b, int n, int lane)
{
    double2 r = make_double2(0, 0);
    for (int i = lane; i < n; i += 32) {
        const float2 t = cconjmul(a[i], b[i]);
        r.x += t.x;
        r.y += t.y;
    }
    for (int s = 16; s >= 1; s >>= 1) {
        r.x += __shfl_xor_sync(0xffffffffu, r.x, s);
        r.y += __shfl_xor_sync(0xffffffffu, r.y, s);
    }
    return r;
}
__device__ __forceinline__ double warp_norm2(const float2 *a, int n, int lane)
{
    double r = 0.0;
    for (int i = lane; i < n; i += 32) r += cabs2(a[i]);
    for (int s = 16; s >= 1; s >>= 1) r += __shfl_xor_sync(0xffffffffu, r, s);
    return r;
}

// Partially pivoted ACA: Z[rows, cols] ~ sum_l u_l v_l^T with u_l stored as the
// row l of U^T (length m) and v_l as row l of V (length n).
//
// Bound by the entry evaluations (a few thousand FP32 instructions each, in dependent
// chains): G::PARTS lanes share one entry (the RWG's four triangle pairs), so that the
// short rows of a block (15 to 64 entries) fill the CTA's warps and a row takes a
// quarter of the chain; the CTA has 64 threads for blocks of up to 32 x 32 (launcher).
// The cross terms of |S_k|_F^2 take one warp per earlier row and no barrier between
// them: FP64 adds run at 2 lanes per clock and SM here, and block-wide sums spent six
// times as many of them.  7,680-unknown sphere (100,000 blocks of 15 x 15): see the
// launcher in assemble().
template <class G>
__global__ void __launch_bounds__(ACA_THREADS)
k_aca(G g, const AcaJob *__restrict__ jobs, float2 *scratch, int32_t *ranks, float tol)
{
    const AcaJob J = jobs[blockIdx.x];
    float2 *UT = scratch + J.off;
    float2 *V = UT + (int64_t)J.kmax * J.m;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    unsigned char *used = smem_raw;           // [m]
    __shared__ float sv[ACA_THREADS / 32];
    __shared__ int si[ACA_THREADS / 32];
    __shared__ double s_nu, s_nv, s_cross[ACA_KCAP];
    const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5;
    const int part = tid % G::PARTS, e0 = tid / G::PARTS, ne = blockDim.x / G::PARTS;
    for (int i = tid; i < J.m; i += blockDim.x) used[i] = 0;
    __syncthreads();
    int k = 0, istar = 0;
    double s2 = 0.0;
    int guard = 0;
    while (k < J.kmax && guard < J.m + J.kmax) {
        ++guard;
        float2 *v = V + (int64_t)k * J.n;
        float2 *u = UT + (int64_t)k * J.m;
        // residual row istar (the lanes of a warp run the same rounds: the parts of an entry are shuffled)
        float best = -1.f;
        int bj = 0;
        for (int j0 = 0; j0 < J.n; j0 += ne) {
            const int j = j0 + e0;
            if (j0 + (tid & ~31) / G::PARTS >= J.n) continue;   // the whole warp is past the row
            const CX<float> z = entry_parts(g, g.perm[J.r0 + istar], g.perm[J.c0 + min(j, J.n - 1)], part);
            if (part != 0 || j >= J.n) continue;
            float2 r = make_float2(z.re, z.im);
            for (int l = 0; l < k; ++l) {
                const float2 p = cmulf(UT[(int64_t)l * J.m + istar], V[(int64_t)l * J.n + j]);
                r.x -= p.x;
                r.y -= p.y;
            }
            v[j] = r;
            const float a = cabs2(r);
            if (a > best) { best = a; bj = j; }
        }
        __syncthreads();
        if (tid == 0) used[istar] = 1;
        float pv;
        int jstar;
        block_argmax(best, bj, sv, si, pv, jstar);
        if (!(pv > 0.f)) {
            int next = -1;
            for (int i = 0; i < J.m; ++i)
                if (!used[i]) { next = i; break; }
            if (next < 0) break;
            istar = next;
            __syncthreads();
            continue;
        }
        const float2 piv = v[jstar];
        __syncthreads();
        const float pn = cabs2(piv);
        const float2 ipiv = make_float2(piv.x / pn, -piv.y / pn);
        for (int j = tid; j < J.n; j += blockDim.x) v[j] = cmulf(v[j], ipiv);
        // residual column jstar
        for (int i0 = 0; i0 < J.m; i0 += ne) {
            const int i = i0 + e0;
            if (i0 + (tid & ~31) / G::PARTS >= J.m) continue;
            const CX<float> z = entry_parts(g, g.perm[J.r0 + min(i, J.m - 1)], g.perm[J.c0 + jstar], part);
            if (part != 0 || i >= J.m) continue;
            float2 c = make_float2(z.re, z.im);
            for (int l = 0; l < k; ++l) {
                const float2 p = cmulf(V[(int64_t)l * J.n + jstar], UT[(int64_t)l * J.m + i]);
                c.x -= p.x;
                c.y -= p.y;
            }
            u[i] = c;
        }
        __syncthreads();
        // norms and the cross terms of |S_k|_F^2: l = k is the new pair itself
        for (int l = k - w; l >= 0; l -= nw) {
            if (l == k) {
                const double nu = warp_norm2(u, J.m, lane), nv = warp_norm2(v, J.n, lane);
                if (lane == 0) { s_nu = nu; s_nv = nv; }
            } else {
                const double2 su = warp_cdot(UT + (int64_t)l * J.m, u, J.m, lane);
                const double2 svv = warp_cdot(V + (int64_t)l * J.n, v, J.n, lane);
                if (lane == 0) s_cross[l] = su.x * svv.x - su.y * svv.y;   // Re(su * svv)
            }
        }
        __syncthreads();
        double cross = 0.0;
        for (int l = 0; l < k; ++l) cross += s_cross[l];
        const double nuv = s_nu * s_nv;
        s2 += 2.0 * cross + nuv;
        ++k;
        if (sqrt(nuv) <= (double)tol * sqrt(fmax(s2, 0.0))) break;
        // next pivot row: largest |u_i| over unused rows
        float bu = -1.f;
        int bi = -1;
        for (int i = tid; i < J.m; i += blockDim.x)
            if (!used[i]) {
                const float a2 = cabs2(u[i]);
                if (a2 > bu) { bu = a2; bi = i; }
            }
        float ov;
        int oi;
        block_argmax(bu, bi < 0 ? 0x7fffffff : bi, sv, si, ov, oi);
        if (ov < 0.f) break;
        istar = oi;
        __syncthreads();
    }
    if (tid == 0) ranks[blockIdx.x] = k;
}

// ------------------------------------------------------------ re-compression ----
// One group of NT threads (a warp, or a CTA of 256 threads for high ranks and long
// blocks) per block.  Orthonormalise the rows of U^T (k x m) and of V (k x n) in place
// by Gram-Schmidt applied twice (R factors in shared memory, FP64), form the core
// C = R_U R_V^T, orthogonalise its columns by one-sided Jacobi rotations
// (C W = [sigma_i w_i]), keep the smallest rank r whose discarded singular values have
// Frobenius norm <= tol * total, and overwrite the rows:
//   U'^T[l] = sum_t (C W)[t][p_l] q_t      V'[l] = sum_t conj(W[t][p_l]) q'_t
// (p = singular values sorted descending), so that U'^T^T V' = Q_U C Q_V^T.
//
// Bound by latency (barriers, FP64 at 2 lanes per clock and SM), so the work is cut to
// need few barriers: the dots of one Gram-Schmidt row run side by side (one warp each),
// and a Jacobi sweep takes its pairs in round-robin steps of k / 2 disjoint pairs
// (Brent & Luk 1985), a group of JG lanes each, instead of k (k - 1) / 2 rotations one
// after another.  A rank of up to 16 takes one warp per block (no CTA barrier at all).
// All blocks of the 7,680-unknown sphere: 59 ms; the pairs one by one, a CTA of 256 threads
// per block and a block-wide sum per dot took 636 ms.
template <int NT> __device__ __forceinline__ void group_sync()
{
    if (NT == 32) __syncwarp();
    else __syncthreads();
}

template <int NT>
__device__ void gram_schmidt_rows(float2 *Q, int k, int len, double2 *Rm /* k x k, Rm[t*k + l] */, double2 *coef,
                                  int tid)
{
    const int lane = tid & 31, w = tid >> 5;
    for (int t = tid; t < k * k; t += NT) Rm[t] = make_double2(0, 0);
    group_sync<NT>();
    for (int l = 0; l < k; ++l) {
        float2 *ql = Q + (int64_t)l * len;
        for (int pass = 0; pass < 2 && l > 0; ++pass) {
            for (int t = w; t < l; t += NT / 32) {
                const double2 s = warp_cdot(Q + (int64_t)t * len, ql, len, lane);
                if (lane == 0) {
                    coef[t] = s;
                    Rm[t * k + l].x += s.x;
                    Rm[t * k + l].y += s.y;
                }
            }
            group_sync<NT>();
            for (int i = tid; i < len; i += NT) {
                float2 v = ql[i];
                for (int t = 0; t < l; ++t) {
                    const float2 q = Q[(int64_t)t * len + i];
                    const float cr = (float)coef[t].x, ci = (float)coef[t].y;
                    v.x -= cr * q.x - ci * q.y;
                    v.y -= cr * q.y + ci * q.x;
                }
                ql[i] = v;
            }
            group_sync<NT>();
        }
        // every warp forms the norm (the same sum)
        const double nrm = sqrt(warp_norm2(ql, len, lane));
        if (tid == 0) Rm[l * k + l] = make_double2(nrm, 0.0);
        const float inv = nrm > 0.0 ? (float)(1.0 / nrm) : 0.f;
        group_sync<NT>();                     // every warp has read the row
        for (int i = tid; i < len; i += NT) {
            ql[i].x *= inv;
            ql[i].y *= inv;
        }
        group_sync<NT>();
    }
}

__device__ __forceinline__ double2 zmul(double2 a, double2 b) { return make_double2(a.x * b.x - a.y * b.y, a.x * b.y + a.y * b.x); }
__device__ __forceinline__ double2 zcmul(double2 a, double2 b) { return make_double2(a.x * b.x + a.y * b.y, a.x * b.y - a.y * b.x); }  // conj(a) b

constexpr int RC_BIG_LEN = 256;   // blocks with a longer side take a CTA (a warp would walk it alone)

// shared bytes of one block of rank up to kc
__host__ __device__ constexpr size_t rc_smem(int kc)
{
    return 4 * (size_t)kc * kc * sizeof(double2) + (((size_t)kc * (sizeof(double2) + sizeof(double) + sizeof(int)) + 3 * sizeof(int) + 15) & ~(size_t)15);
}

// WPC blocks per CTA, NT threads each; kc = the largest rank of the launch
template <int NT, int WPC, int JG>
__global__ void __launch_bounds__(NT * WPC)
k_recompress(const AcaJob *__restrict__ jobs, int njobs, float2 *scratch, int32_t *ranks, float tol, int kc)
{
    const int sub = threadIdx.x / NT, tid = threadIdx.x % NT;
    const int job = blockIdx.x * WPC + sub;
    if (job >= njobs) return;                 // whole warps (NT = 32) or the CTA
    const AcaJob J = jobs[job];
    const int k = ranks[job];
    if (k <= 1) return;
    float2 *UT = scratch + J.off;
    float2 *V = UT + (int64_t)J.kmax * J.m;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    double2 *Ru = reinterpret_cast<double2 *>(smem_raw + sub * rc_smem(kc));   // k x k
    double2 *Rv = Ru + k * k;                              // k x k
    double2 *C = Rv + k * k;                               // k x k, column-major C[col*k + row]
    double2 *W = C + k * k;                                // k x k, column-major
    double2 *coef = W + k * k;                             // k
    double *sig = reinterpret_cast<double *>(coef + k);    // k
    int *order = reinterpret_cast<int *>(sig + k);         // k
    int *flags = order + k;                                // rotated in this sweep (two, alternating); kept rank
    gram_schmidt_rows<NT>(UT, k, J.m, Ru, coef, tid);
    gram_schmidt_rows<NT>(V, k, J.n, Rv, coef, tid);
    // C = Ru Rv^T (both upper triangular, Rm[t*k + l] = R[t][l])
    for (int e = tid; e < k * k; e += NT) {
        const int row = e % k, col = e / k;
        double2 s = make_double2(0, 0);
        for (int t = max(row, col); t < k; ++t) {
            const double2 p = zmul(Ru[row * k + t], Rv[col * k + t]);
            s.x += p.x; s.y += p.y;
        }
        C[col * k + row] = s;
        W[col * k + row] = make_double2(row == col ? 1.0 : 0.0, 0.0);
    }
    if (tid < 2) flags[tid] = 0;
    group_sync<NT>();
    // one-sided Jacobi on the columns of C: step s of a sweep pairs (k2 - 1, s) and
    // (s + i, s - i) mod (k2 - 1), i = 1 .. k2/2 - 1, k2 = k rounded up to even (a pair with
    // the column k that is not there is skipped); JG lanes form a pair's 2x2 Gram entries
    // and rotate its rows
    const int k2 = (k + 1) & ~1, jl = tid % JG;
    for (int sweep = 0; sweep < 20; ++sweep) {
        if (tid == 0) flags[(sweep + 1) & 1] = 0;
        for (int s = 0; s < k2 - 1; ++s) {
            for (int i0 = 0; i0 < k2 / 2; i0 += NT / JG) {
                const int i = i0 + tid / JG;
                int p = k2 - 1, q = s;
                if (i > 0) { p = (s + i) % (k2 - 1); q = (s + k2 - 1 - i) % (k2 - 1); }
                if (p > q) { const int t = p; p = q; q = t; }
                const bool on = i < k2 / 2 && q < k;
                double al = 0, be = 0, gr = 0, gi = 0;
                if (on)
                    for (int t = jl; t < k; t += JG) {
                        const double2 cp = C[p * k + t], cq = C[q * k + t];
                        al += cp.x * cp.x + cp.y * cp.y;
                        be += cq.x * cq.x + cq.y * cq.y;
                        gr += cp.x * cq.x + cp.y * cq.y;
                        gi += cp.x * cq.y - cp.y * cq.x;
                    }
#pragma unroll
                for (int o = JG / 2; o >= 1; o >>= 1) {
                    al += __shfl_xor_sync(0xffffffffu, al, o);
                    be += __shfl_xor_sync(0xffffffffu, be, o);
                    gr += __shfl_xor_sync(0xffffffffu, gr, o);
                    gi += __shfl_xor_sync(0xffffffffu, gi, o);
                }
                const double g2 = gr * gr + gi * gi;
                if (on && g2 > 1e-24 * (al * be) && g2 > 0.0) {
                    const double gabs = sqrt(g2);
                    const double zeta = (be - al) / (2.0 * gabs);
                    const double tt = (zeta >= 0 ? 1.0 : -1.0) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
                    const double c = 1.0 / sqrt(1.0 + tt * tt);
                    const double sg = c * tt / gabs;
                    const double2 sv = make_double2(sg * gr, sg * gi);   // s = |s| gamma / |gamma|
                    for (int t = jl; t < 2 * k; t += JG) {
                        double2 *M = t < k ? C : W;
                        const int r = t < k ? t : t - k;
                        const double2 a = M[p * k + r], b = M[q * k + r];
                        // [a b] <- [a b] [[c, s], [-conj(s), c]]
                        const double2 csb = zcmul(sv, b);   // conj(s) b
                        const double2 sa = zmul(sv, a);
                        M[p * k + r] = make_double2(c * a.x - csb.x, c * a.y - csb.y);
                        M[q * k + r] = make_double2(sa.x + c * b.x, sa.y + c * b.y);
                    }
                    if (jl == 0) flags[sweep & 1] = 1;
                }
            }
            group_sync<NT>();
        }
        const int rot = flags[sweep & 1];
        group_sync<NT>();
        if (!rot) break;
    }
    // singular values and truncation
    for (int l = tid; l < k; l += NT) {
        double a = 0;
        for (int t = 0; t < k; ++t) a += C[l * k + t].x * C[l * k + t].x + C[l * k + t].y * C[l * k + t].y;
        sig[l] = sqrt(a);
    }
    group_sync<NT>();
    if (tid == 0) {
        for (int l = 0; l < k; ++l) order[l] = l;
        for (int a = 1; a < k; ++a) {   // insertion sort, descending
            const int key = order[a];
            int b = a - 1;
            while (b >= 0 && sig[order[b]] < sig[key]) { order[b + 1] = order[b]; --b; }
            order[b + 1] = key;
        }
        double total = 0;
        for (int l = 0; l < k; ++l) total += sig[l] * sig[l];
        double tail = total;
        int r = k;
        for (int l = 0; l < k; ++l) {   // tail = sum of sig[order[l..]]^2
            if (l >= 1 && sqrt(fmax(tail, 0.0)) <= tol * sqrt(total)) { r = l; break; }
            tail -= sig[order[l]] * sig[order[l]];
        }
        if (r < 1) r = 1;
        flags[2] = r;
    }
    group_sync<NT>();
    const int r = flags[2];
    // rows of U'^T and V' : each thread owns one position and transforms its k-vector
    for (int side = 0; side < 2; ++side) {
        float2 *Q = side == 0 ? UT : V;
        const int len = side == 0 ? J.m : J.n;
        for (int i = tid; i < len; i += NT) {
            float2 qv[ACA_KCAP];
            for (int t = 0; t < k; ++t) qv[t] = Q[(int64_t)t * len + i];
            for (int l = 0; l < r; ++l) {
                const int pl = order[l];
                double2 s = make_double2(0, 0);
                for (int t = 0; t < k; ++t) {
                    const double2 q = make_double2(qv[t].x, qv[t].y);
                    const double2 m = side == 0 ? C[pl * k + t] : make_double2(W[pl * k + t].x, -W[pl * k + t].y);
                    const double2 p = zmul(m, q);
                    s.x += p.x; s.y += p.y;
                }
                Q[(int64_t)l * len + i] = make_float2((float)s.x, (float)s.y);
            }
        }
    }
    if (tid == 0) ranks[job] = r;
}

// re-compression of the blocks jb (ranks rb, on the device), all of rank at most kc
inline hm_status launch_recompress(const AcaJob *jb, int n, float2 *scr, int32_t *rb, float tol, int kc, bool big,
                                   cudaStream_t s)
{
    constexpr int WPC = 4;
    auto go = [&](auto kern, int wpc, int threads) -> hm_status {
        const size_t sm = wpc * rc_smem(kc);
        HM_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm));
        kern<<<(unsigned)((n + wpc - 1) / wpc), threads, sm, s>>>(jb, n, scr, rb, tol, kc);
        return HM_OK;
    };
    hm_status st;
    if (kc <= 8 && !big) st = go(k_recompress<32, WPC, 8>, WPC, 32 * WPC);
    else if (kc <= 16 && !big) st = go(k_recompress<32, WPC, 4>, WPC, 32 * WPC);
    else st = go(k_recompress<RC_THREADS, 1, 8>, 1, RC_THREADS);
    if (st != HM_OK) return st;
    HM_CUDA(cudaGetLastError());
    return HM_OK;
}

// copy rank-r factors from the ACA scratch into the padded pool
struct PackJob {
    int64_t src;     // scratch offset (U^T kmax x m, V kmax x n)
    int64_t dst;     // pool offset (U^T r x pm, V r x pn)
    int32_t r0, c0;  // tree positions (true)
    int32_t pr0, pc0;// padded positions
    int32_t m, n, pm, pn, kmax, r;
};

__global__ void k_pack_far(const PackJob *__restrict__ jobs, const float2 *__restrict__ scratch,
                           const int32_t *__restrict__ ptree, float2 *pool)
{
    const PackJob J = jobs[blockIdx.x];
    const int64_t nu = (int64_t)J.r * J.pm, nv = (int64_t)J.r * J.pn;
    for (int64_t e = threadIdx.x; e < nu + nv; e += blockDim.x) {
        float2 v = make_float2(0.f, 0.f);
        if (e < nu) {
            const int l = (int)(e / J.pm), pi = (int)(e - (int64_t)l * J.pm);
            const int tp = ptree[J.pr0 + pi];
            if (tp >= 0) v = scratch[J.src + (int64_t)l * J.m + (tp - J.r0)];
        } else {
            const int64_t e2 = e - nu;
            const int l = (int)(e2 / J.pn), pj = (int)(e2 - (int64_t)l * J.pn);
            const int tp = ptree[J.pc0 + pj];
            if (tp >= 0) v = scratch[J.src + (int64_t)J.kmax * J.m + (int64_t)l * J.n + (tp - J.c0)];
        }
        pool[J.dst + e] = v;
    }
}

// ------------------------------------------------------------ host side ---------
struct HostTree {
    std::vector<std::vector<std::pair<int64_t, int64_t>>> levels;   // (offset, size) per depth
    std::vector<std::vector<std::vector<int>>> children;           // per depth
    std::vector<std::vector<std::array<double, 6>>> box;           // lo[3], hi[3]
    std::vector<int64_t> perm;
    int depth = 0;
};


// bisect idx along the longest axis of the bounding box of its centres; ties in
// the axis go to the lower axis; sort key (coordinate, original index); cut at n/2
void bisect(const std::vector<int64_t> &idx, const std::vector<double> &cen, std::vector<int64_t> &a,
            std::vector<int64_t> &b)
{
    double lo[3] = {INFINITY, INFINITY, INFINITY}, hi[3] = {-INFINITY, -INFINITY, -INFINITY};
    for (int64_t v : idx)
        for (int d = 0; d < 3; ++d) {
            lo[d] = std::min(lo[d], cen[3 * v + d]);
            hi[d] = std::max(hi[d], cen[3 * v + d]);
        }
    int axis = 0;
    double best = hi[0] - lo[0];
    for (int d = 1; d < 3; ++d)
        if (hi[d] - lo[d] > best) { best = hi[d] - lo[d]; axis = d; }
    std::vector<int64_t> s = idx;
    std::sort(s.begin(), s.end(), [&](int64_t x, int64_t y) {
        const double cx = cen[3 * x + axis], cy = cen[3 * y + axis];
        return cx < cy || (cx == cy && x < y);
    });
    const size_t h = s.size() / 2;
    a.assign(s.begin(), s.begin() + h);
    b.assign(s.begin() + h, s.end());
}

hm_status build_tree(const std::vector<double> &cen, const std::vector<double> &blo, const std::vector<double> &bhi,
                     int64_t N, int leaf_size, int arity, HostTree &T)
{
    const int splits = arity == 2 ? 1 : arity == 4 ? 2 : 3;
    std::vector<std::vector<int64_t>> clusters(1);
    clusters[0].resize(N);
    std::iota(clusters[0].begin(), clusters[0].end(), 0);
    std::vector<std::vector<std::vector<int64_t>>> lv{clusters};
    while (true) {
        size_t mx = 0;
        for (auto &c : clusters) mx = std::max(mx, c.size());
        if ((int64_t)mx <= leaf_size) break;
        std::vector<std::vector<int64_t>> nxt;
        std::vector<std::vector<int>> ch;
        for (auto &c : clusters) {
            std::vector<std::vector<int64_t>> parts{c};
            for (int s = 0; s < splits; ++s) {
                std::vector<std::vector<int64_t>> np;
                for (auto &p : parts) {
                    std::vector<int64_t> a, b;
                    bisect(p, cen, a, b);
                    np.push_back(std::move(a));
                    np.push_back(std::move(b));
                }
                parts.swap(np);
            }
            std::vector<int> kids;
            for (auto &p : parts) {
                if (p.empty()) return fail(HM_ERR_ARG, "leaf_size too small for this arity: a cluster would be empty");
                kids.push_back((int)nxt.size());
                nxt.push_back(std::move(p));
            }
            ch.push_back(kids);
        }
        T.children.push_back(ch);
        clusters.swap(nxt);
        lv.push_back(clusters);
    }
    T.depth = (int)lv.size() - 1;
    T.perm.clear();
    for (auto &c : clusters) T.perm.insert(T.perm.end(), c.begin(), c.end());
    std::vector<int64_t> pos(N);
    for (int64_t p = 0; p < N; ++p) pos[T.perm[p]] = p;
    for (auto &cl : lv) {
        std::vector<std::pair<int64_t, int64_t>> L;
        std::vector<std::array<double, 6>> B;
        for (auto &c : cl) {
            int64_t mn = N;
            std::array<double, 6> bx{INFINITY, INFINITY, INFINITY, -INFINITY, -INFINITY, -INFINITY};
            for (int64_t v : c) {
                mn = std::min(mn, pos[v]);
                for (int d = 0; d < 3; ++d) {
                    bx[d] = std::min(bx[d], blo[3 * v + d]);
                    bx[3 + d] = std::max(bx[3 + d], bhi[3 * v + d]);
                }
            }
            L.push_back({mn, (int64_t)c.size()});
            B.push_back(bx);
        }
        T.levels.push_back(L);
        T.box.push_back(B);
    }
    return HM_OK;
}

bool admissible(const HostTree &T, int d, int t, int s, double c)
{
    const auto &a = T.box[d][t], &b = T.box[d][s];
    double g2 = 0, da = 0, db = 0;
    for (int x = 0; x < 3; ++x) {
        const double gap = std::max(0.0, std::max(b[x] - a[3 + x], a[x] - b[3 + x]));
        g2 = g2 + gap * gap;
        const double ea = a[3 + x] - a[x], eb = b[3 + x] - b[x];
        da = da + ea * ea;
        db = db + eb * eb;
    }
    const double dist = std::sqrt(g2);
    return dist > 0.0 && dist >= c * std::min(std::sqrt(da), std::sqrt(db));
}

void partition(const HostTree &T, double c, int d, int t, int s, std::vector<std::pair<int, int>> &near,
               std::map<int, std::vector<std::pair<int, int>>> &far)
{
    if (t != s && admissible(T, d, t, s, c)) {
        far[d].push_back({t, s});
        return;
    }
    if (d == T.depth) {
        if (t != s) near.push_back({t, s});
        return;
    }
    for (int ct : T.children[d][t])
        for (int cs : T.children[d][s]) {
            if (t == s && ct > cs) continue;
            partition(T, c, d + 1, ct, cs, near, far);
        }
}

template <class T> hm_status up(hm_matrix h, T **dst, const std::vector<T> &src, cudaStream_t s)
{
    hm_status st = dev_alloc(h, (void **)dst, std::max<size_t>(1, src.size()) * sizeof(T));
    if (st != HM_OK) return st;
    if (!src.empty()) HM_CUDA(cudaMemcpyAsync(*dst, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, s));
    return HM_OK;
}

struct TmpBuffers {
    std::vector<void *> ptrs;
    ~TmpBuffers() { for (void *p : ptrs) cudaFree(p); }
    template <class T> hm_status up(T **dst, const std::vector<T> &src, cudaStream_t s)
    {
        void *p = nullptr;
        const size_t bytes = std::max<size_t>(1, src.size()) * sizeof(T);
        HM_CUDA(cudaMalloc(&p, bytes));
        ptrs.push_back(p);
        *dst = (T *)p;
        if (!src.empty()) HM_CUDA(cudaMemcpyAsync(p, src.data(), src.size() * sizeof(T), cudaMemcpyHostToDevice, s));
        return HM_OK;
    }
    hm_status alloc(void **dst, size_t bytes)
    {
        HM_CUDA(cudaMalloc(dst, std::max<size_t>(bytes, 16)));
        ptrs.push_back(*dst);
        return HM_OK;
    }
};

// the middle of the points' bounding box
inline std::array<double, 3> middle(const std::vector<double> &v)
{
    std::array<double, 3> c{};
    for (int d = 0; d < 3; ++d) {
        double lo = v[d], hi = v[d];
        for (size_t i = d; i < v.size(); i += 3) { lo = std::min(lo, v[i]); hi = std::max(hi, v[i]); }
        c[d] = 0.5 * lo + 0.5 * hi;
    }
    return c;
}

// points relative to c, each coordinate as the pair (hi, lo) of floats, hi the nearest float, lo the
// nearest to the rest: 49 bits of the object's size, wherever it lies (only differences of two such
// points are used)
inline std::vector<float2> float_pairs(const std::vector<double> &v, const std::array<double, 3> &c)
{
    std::vector<float2> r(v.size());
    for (size_t i = 0; i < v.size(); ++i) {
        const double x = v[i] - c[i % 3];
        r[i].x = (float)x;
        r[i].y = (float)(x - (double)r[i].x);
    }
    return r;
}

// Host description of the unknowns of one basis: the point each unknown is
// sorted by in the tree and its support box, plus what the operator keeps for
// plane-wave excitation (b_m = sum over the two sides of ucoef * sum_q w_q
// (r_q - v) . p exp(-jk k . r_q) over the side's cell).
struct BasisData {
    int64_t N = 0;
    std::vector<double> cen, blo, bhi;   // N x 3 each
    int nq = 0;                          // quadrature points per cell
    std::vector<double> qw;              // nq weights (sum 1)
    std::vector<double> qpd;             // n_cell x nq x 3 points
    std::vector<double> vtx;             // n_vert x 3
    std::vector<int32_t> ucell, ufree;   // N x 2: cell and free vertex of each side (-1: no side)
    std::vector<double> ucoef;           // N x 2
};

// Tree, partition, packed layout, far-field ACA + re-compression and near fill
// for the basis geometry g (all device pointers set except g.perm).
template <class G>
hm_status assemble(BasisData &B, G g, const hm_build_opts *o, TmpBuffers &tmp, cudaStream_t s, hm_matrix *out)
{
    const int64_t N = B.N;
    HostTree T;
    hm_status st = build_tree(B.cen, B.blo, B.bhi, N, o->leaf_size, o->arity, T);
    if (st != HM_OK) return st;
    std::vector<std::pair<int, int>> near;
    std::map<int, std::vector<std::pair<int, int>>> farp;
    partition(T, o->adm, 0, 0, 0, near, farp);

    hm_matrix h = new hm_matrix_s();
    struct Guard { hm_matrix h; bool keep = false; ~Guard() { if (!keep && h) hm_destroy(h); } } guard{h};
    h->N = N;
    h->perm = T.perm;
    h->n_leaves = (int64_t)T.levels[T.depth].size();
    h->leaf_off.resize(h->n_leaves + 1);
    for (int64_t i = 0; i < h->n_leaves; ++i) h->leaf_off[i] = T.levels[T.depth][i].first;
    h->leaf_off[h->n_leaves] = N;
    h->has_fp64 = o->keep_fp64 != 0;
    if ((st = finalize_layout(h, s)) != HM_OK) return st;
    h->depth = T.depth;

    std::vector<int32_t> perm32(T.perm.begin(), T.perm.end());
    int32_t *d_perm = nullptr;
    if ((st = tmp.up(&d_perm, perm32, s)) != HM_OK) return st;
    g.perm = d_perm;

    // ---- far blocks: ACA + re-compression into scratch
    const int max_level_keep = o->levels < 0 ? 1 << 20 : o->levels;
    struct FarRec { int level; int64_t r0, m, c0, n; };
    std::vector<FarRec> fars;
    for (auto &kv : farp) {
        const int lev = T.depth - kv.first + 1;
        if (lev > max_level_keep) continue;
        for (auto &pr : kv.second) {
            const auto &a = T.levels[kv.first][pr.first], &b = T.levels[kv.first][pr.second];
            fars.push_back({lev, a.first, a.second, b.first, b.second});
        }
    }
    std::vector<AcaJob> aj(fars.size());
    int64_t scr = 0;
    for (size_t b = 0; b < fars.size(); ++b) {
        const int kmax = (int)std::min<int64_t>(ACA_KCAP, std::min(fars[b].m, fars[b].n));
        aj[b] = {scr, (int32_t)fars[b].r0, (int32_t)fars[b].c0, (int32_t)fars[b].m, (int32_t)fars[b].n, kmax, 0};
        scr += (int64_t)kmax * (fars[b].m + fars[b].n);
    }
    float2 *d_scr = nullptr;
    int32_t *d_ranks = nullptr;
    AcaJob *d_aj = nullptr;
    std::vector<int32_t> ranks(fars.size(), 0);
    if (!fars.empty()) {
        if ((st = tmp.alloc((void **)&d_scr, sizeof(float2) * scr)) != HM_OK) return st;
        if ((st = tmp.alloc((void **)&d_ranks, sizeof(int32_t) * fars.size())) != HM_OK) return st;
        if ((st = tmp.up(&d_aj, aj, s)) != HM_OK) return st;
        int64_t maxm = 0;
        for (auto &j : aj) maxm = std::max<int64_t>(maxm, j.m);
        // two warps a block up to 32 x 32 (its rows are 15 to 32 entries of PARTS lanes), four above
        const int at = maxm <= 32 ? 64 : ACA_THREADS;
        k_aca<G><<<(unsigned)fars.size(), at, maxm, s>>>(g, d_aj, d_scr, d_ranks, (float)o->aca_tol);
        HM_CUDA(cudaGetLastError());
        HM_CUDA(cudaMemcpyAsync(ranks.data(), d_ranks, sizeof(int32_t) * fars.size(), cudaMemcpyDeviceToHost, s));
        HM_CUDA(cudaStreamSynchronize(s));
        // re-compression, launched per rank bucket so that shared memory fits the bucket, blocks
        // of a long side apart; one read-back of the new ranks at the end
        const int bounds[] = {8, 16, 32, ACA_KCAP};
        std::vector<AcaJob> jb;
        std::vector<int32_t> rb;
        std::vector<size_t> where;
        struct Launch { size_t first, n; int kc; bool big; };
        std::vector<Launch> ls;
        int lo = 1;
        for (int bk : bounds) {
            for (bool big : {false, true}) {
                const size_t first = where.size();
                for (size_t b = 0; b < fars.size(); ++b)
                    if (ranks[b] > lo && ranks[b] <= bk && (std::max(aj[b].m, aj[b].n) > RC_BIG_LEN) == big) {
                        jb.push_back(aj[b]);
                        rb.push_back(ranks[b]);
                        where.push_back(b);
                    }
                if (where.size() > first) ls.push_back({first, where.size() - first, bk, big});
            }
            lo = bk;
        }
        if (!where.empty()) {
            AcaJob *d_jb = nullptr;
            int32_t *d_rb = nullptr;
            if ((st = tmp.up(&d_jb, jb, s)) != HM_OK) return st;
            if ((st = tmp.up(&d_rb, rb, s)) != HM_OK) return st;
            for (const Launch &l : ls)
                if ((st = launch_recompress(d_jb + l.first, (int)l.n, d_scr, d_rb + l.first, (float)o->aca_tol, l.kc,
                                            l.big, s)) != HM_OK)
                    return st;
            HM_CUDA(cudaMemcpyAsync(rb.data(), d_rb, sizeof(int32_t) * rb.size(), cudaMemcpyDeviceToHost, s));
            HM_CUDA(cudaStreamSynchronize(s));
            for (size_t q = 0; q < where.size(); ++q) ranks[where[q]] = rb[q];
        }
    }

    // ---- pool layout: near blocks (level 1) then far blocks, by level
    std::map<int64_t, int64_t> leaf_start, leaf_end;
    for (int64_t i = 0; i < h->n_leaves; ++i) {
        leaf_start[h->leaf_off[i]] = i;
        leaf_end[h->leaf_off[i + 1]] = i;
    }
    auto padded = [&](int64_t r0, int64_t m, int64_t &pr0, int64_t &pm) {
        const int64_t a = leaf_start.at(r0), b = leaf_end.at(r0 + m);
        pr0 = h->pleaf_off[a];
        pm = h->pleaf_off[b + 1] - pr0;
    };
    int64_t pool = 0;
    std::vector<FillJob> fj, fs;   // near jobs, self jobs
    int64_t flat = 0, flat_self = 0;
    for (auto &pr : near) {
        const auto &a = T.levels[T.depth][pr.first], &b = T.levels[T.depth][pr.second];
        Item it{};
        int64_t pr0, pm, pc0, pn;
        padded(a.first, a.second, pr0, pm);
        padded(b.first, b.second, pc0, pn);
        it.off = pool; it.row0 = (int32_t)pr0; it.col0 = (int32_t)pc0;
        it.m = (int32_t)a.second; it.n = (int32_t)b.second; it.k = 0;
        fj.push_back({it.off, flat, (int32_t)a.first, (int32_t)b.first, it.m, it.n, (int32_t)even(it.n), 0});
        flat += (int64_t)it.m * it.n;
        pool += item_elems(it);
        LevelList &L = h->levels[1];
        L.items.push_back(it); L.true_m.push_back(it.m); L.true_n.push_back(it.n);
        L.elems += item_elems(it); L.n_dense++;
        L.alg_elems += (int64_t)it.m * it.n;
    }
    std::vector<PackJob> pj;
    int max_level = 1, max_rank = 0;
    for (size_t b = 0; b < fars.size(); ++b) {
        const FarRec &f = fars[b];
        Item it{};
        int64_t pr0, pm, pc0, pn;
        padded(f.r0, f.m, pr0, pm);
        padded(f.c0, f.n, pc0, pn);
        it.off = pool; it.row0 = (int32_t)pr0; it.col0 = (int32_t)pc0;
        it.m = (int32_t)pm; it.n = (int32_t)pn; it.k = ranks[b];
        if (it.k < 1) continue;   // an exactly zero block
        pj.push_back({aj[b].off, it.off, (int32_t)f.r0, (int32_t)f.c0, (int32_t)pr0, (int32_t)pc0, (int32_t)f.m,
                      (int32_t)f.n, (int32_t)pm, (int32_t)pn, aj[b].kmax, it.k});
        pool += item_elems(it);
        LevelList &L = h->levels[f.level];
        L.items.push_back(it); L.true_m.push_back((int32_t)f.m); L.true_n.push_back((int32_t)f.n);
        L.elems += item_elems(it); L.n_lowrank++;
        L.alg_elems += (int64_t)it.k * (f.m + f.n);
        max_level = std::max(max_level, f.level);
        max_rank = std::max(max_rank, it.k);
    }
    // self blocks (complex128, upper half + mirror)
    for (int64_t i = 0; i < h->n_leaves; ++i) {
        const int64_t n = h->leaf_off[i + 1] - h->leaf_off[i];
        fs.push_back({h->self_off[i], flat_self, (int32_t)h->leaf_off[i], (int32_t)h->leaf_off[i], (int32_t)n,
                      (int32_t)n, 0, 1});
        flat_self += n * (n + 1) / 2;
    }
    h->pool_elems = pool;
    h->n_levels = max_level;
    h->max_rank = max_rank;
    if ((st = dev_alloc(h, (void **)&h->d_pool32, sizeof(float2) * std::max<int64_t>(pool, 1))) != HM_OK) return st;
    HM_CUDA(cudaMemsetAsync(h->d_pool32, 0, sizeof(float2) * std::max<int64_t>(pool, 1), s));
    if ((st = dev_alloc(h, (void **)&h->d_self64, sizeof(double2) * h->self_elems)) != HM_OK) return st;
    FillJob *d_fj = nullptr, *d_fs = nullptr;
    if ((st = tmp.up(&d_fj, fj, s)) != HM_OK) return st;
    if ((st = tmp.up(&d_fs, fs, s)) != HM_OK) return st;
    if (flat > 0) {
      if constexpr (G::BLOCK_FILL) {   // the basis fills whole blocks (its element integrals serve many entries)
        if ((st = g.fill_near(fj, h->d_pool32, tmp, s)) != HM_OK) return st;
      } else {
        const int grid = (int)std::min<int64_t>((flat + 255) / 256, 152 * 64);
        k_fill<G, false><<<grid, 256, 0, s>>>(g, d_fj, (int)fj.size(), flat, h->d_pool32, h->d_self64);
        HM_CUDA(cudaGetLastError());
      }
    }
    if (flat_self > 0) {
        const int grid = (int)std::min<int64_t>((flat_self + 255) / 256, 152 * 64);
        k_fill<G, true><<<grid, 256, 0, s>>>(g, d_fs, (int)fs.size(), flat_self, h->d_pool32, h->d_self64);
        HM_CUDA(cudaGetLastError());
    }
    if (!pj.empty()) {
        std::vector<int32_t> ptree(h->pN, -1);
        for (int64_t i = 0; i < h->n_leaves; ++i)
            for (int64_t p = h->leaf_off[i]; p < h->leaf_off[i + 1]; ++p)
                ptree[h->pleaf_off[i] + (p - h->leaf_off[i])] = (int32_t)p;
        int32_t *d_ptree = nullptr;
        PackJob *d_pj = nullptr;
        if ((st = tmp.up(&d_ptree, ptree, s)) != HM_OK) return st;
        if ((st = tmp.up(&d_pj, pj, s)) != HM_OK) return st;
        k_pack_far<<<(unsigned)pj.size(), 256, 0, s>>>(d_pj, d_scr, d_ptree, h->d_pool32);
        HM_CUDA(cudaGetLastError());
    }
    if (h->has_fp64) {   // complex128 copy of the same (complex64-filled) blocks for the FP64 path
        if ((st = dev_alloc(h, (void **)&h->d_pool64, sizeof(double2) * std::max<int64_t>(pool, 1))) != HM_OK)
            return st;
        launch_convert_f32_to_f64(h->d_pool32, h->d_pool64, std::max<int64_t>(pool, 1), s);
    }
    if ((st = prepare_partials(h, s)) != HM_OK) return st;
    if ((st = upload_item_lists(h, s)) != HM_OK) return st;
    // geometry kept for the plane-wave excitation
    if ((st = up(h, &h->d_qpd, B.qpd, s)) != HM_OK || (st = up(h, &h->d_vtx, B.vtx, s)) != HM_OK ||
        (st = up(h, &h->d_ucell, B.ucell, s)) != HM_OK || (st = up(h, &h->d_ufree, B.ufree, s)) != HM_OK ||
        (st = up(h, &h->d_ucoef, B.ucoef, s)) != HM_OK || (st = up(h, &h->d_rhs_w, B.qw, s)) != HM_OK)
        return st;
    h->rhs_nq = B.nq;
    h->has_mesh = true;
    h->wavenumber = g.k;
    HM_CUDA(cudaStreamSynchronize(s));
    guard.keep = true;
    *out = h;
    return HM_OK;
}

} // namespace
} // namespace hm
