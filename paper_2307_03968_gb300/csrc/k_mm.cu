// Block products for many right-hand sides on the matrix instructions (arxiv 2307.03968
// eqs. 6 and 8 with the half storage of §III, blocks of up to 64 x 64 and rank 32):
//     Z_I += B X_J, Z_J += B^T X_I;   Z_I += U (V X_J), Z_J += V^T (U^T X_I)
// as two dense products over lists (hm_lists.h, build_mm_lists): stage 1, per input cluster,
// T = W X_J with the rank rows of all its low-rank products stacked; then per output
// cluster [B_1 B_2 .. Y_1 Y_2 ..] [X; X; .. T_1; T_2; ..], the ranks concatenated along K, so that
// neither a rank nor a block is padded to an instruction's shape (only the 16 of a chunk
// and the 8 of a cluster's outputs).
//
// Why mma.sync m16n8k16 with 16-bit operands.  It runs at twice the rate of TF32 (measured,
// registers only: 606 against 302 TFLOP/s; the tcgen05 kernel of k_mrhs_tc.cu, 1952 TFLOP/s in
// bf16, reaches 28 % of its TF32 roof on the hand-offs of its operand pipeline), and a call of 4
// to 64 right-hand sides fills its tiles of 16, which a tile of 128 does not.  BF16 parts for the
// FP32 product, FP16 digits for the residual.
//
// Operand streams.  The first call repacks the blocks (k_mm_pack_*): for each chunk of 16 K and
// tile of 8 outputs the 128 values in the order the lanes of the instruction take them, FP32,
// scaled, both directions of every block: twice the blocks' bytes.  A unit's blocks are then
// one contiguous stream, copied with a few cp.async a thread, and what is left beside the
// instructions is the split into parts or digits in registers.  (Gathered from the blocks
// in place, by rows and by columns, the same kernels spent 500 instructions on 24 products:
// 0.60 ms instead of 0.31 for 16 right-hand sides of the 12,600-unknown cube.)
//
// Measured (GB300): a product of the 30,720-unknown sphere with 181 right-hand sides 10.2 ms
// (the tcgen05 kernels, of 3xTF32 accuracy, 8.0), with 64 of them 3.4 (SIMT chunks of 16: 11.8),
// with 16 1.0 (3.0); 16 right-hand sides of the 12,600-unknown cube 0.53 ms (0.69); hm_residual
// with the FP64-class sums of the 181 34 ms (owner kernel on the FP32 pipes: 72) and of the 16 1.7 ms
// (2.4).
//
// Right-hand sides are the instruction's M, so an accumulator pair of stage 1 is, in place,
// an operand pair of the output stage (its K are the W rows): T is stored in operand layout.
// Operand tile of 16 right-hand sides x 16 K: one plane per part or digit (product: re 1..3, im
// 1..3; residual: re 1..5, im 1..5), each 4 registers x 32 words; word t * 8 + g of
// register r is the pair of K 2t, 2t + 1 (+ 8 for r >= 2) of right-hand side g (+ 8 for odd r):
// what lane (g, t) holds, and 32 bytes per t, so that stage 1 writes whole sectors.
//
// Scales (powers of two, exact).  The streams hold W row l times 2^et(l), |W_l|_1 <= 1 with it, and Y
// row l (dense blocks: the block) times 2^(E - et(l)), E per output cluster the largest that keeps all
// its entries at most 1 (k_mm_prep, once per operator).  The product takes x times 2^-ex, ex per
// right-hand side (k_mm_max).  The residual's digits have scales of their own: of x per chunk of 16
// and right-hand side (k_mm_split), of T per chunk and right-hand side, from the x below it
// (k_mm_tscale), and of the blocks per chunk and row (packed beside the streams); every chunk's sums are
// brought to one unit where they leave the tensor core.  Scales are exponents, never cut off at a
// float's range (times_pow2, pow2x): one that is would be missing from the sum's factor.
//
// Product: a = a1 + a2 + a3, three BF16 parts of 8 bits, an FP32 number exactly (the last bits of
// one below 2^-109 of the scale apart): a1 b1 + a1 b2 + a2 b1 + a1 b3 + a2 b2 + a3 b1, the three
// left out are below 2^-25 of a b and of either sign, the parts being rounded to nearest (cut off,
// they leave out terms of one sign: the refined solve of a 3,001-unknown import erred by 2.7e-7, so by
// 1.8e-7, with the FP32 kernels by 1.9e-7).  BF16 has FP32's exponents, so a small operand keeps its bits
// beside a large one; two FP16 halves (22 bits, three products, 6.4 ms for those 181) lose them
// below 2^-17 of the scale: entries at 2^-30 came out to 1e-3.  The tensor core truncates its FP32 sums,
// so each chunk's sums start from zero and join the running sum in FP32; 32 chunks in the tensor
// core instead of one took 6 % less time and erred by 1e-6 of |A x| (5e-6 in that solve).  What is left
// is the mean of the truncation, 5e-9 of |A x|; adding every second chunk times 1 + 2^-23 takes it back
// (1.4e-7) but makes exact products inexact, so it is not done.
//
// FP64-class residual: a = 2^-8 d1 + 2^-17 d2 + 2^-26 d3 + 2^-35 d4 + 2^-44 r, the digits integers of at
// most 2^8 (a unit or two more for T), r a FP16 of at most 2^8: 48 bits below the scale, exact for every FP32
// a >= 2^-24 of it (integer digits on a common grid follow Ozaki, Ogita, Oishi & Rump 2012).
// Fifteen products, those of digits i and j with i + j <= 6, in five sums of weights 2^-16, 2^-25,
// 2^-34, 2^-43, 2^-52; the dropped ones are below 2^-45.  The first four are sums of integers, of at
// most 4 x 32 x 2^16 = 2^23 in a chunk, exact in the tensor core's truncating FP32 sums; each chunk then
// joins a double-float sum.  Against 64 bits, in units of the sum of the moduli: 2^-44 rms (the
// owner kernel on the FP32 pipes 2^-42), 2^-40 to 2^-42 for vectors graded over 2^-30 (2^-39 to 2^-41).
// Four digits of 38 bits on one scale per right-hand side, drained every 4 chunks, took a quarter
// less time and erred by 2^-41, graded by 2^-33.
#include "k_dot2.cuh"

#include <cuda_fp16.h>

#include <algorithm>

namespace hm {
namespace {

using namespace kc;
using namespace dot2;

constexpr int MMW = 8;                    // warps per CTA
constexpr int MM_PLANE = 128;             // words of one plane of an operand tile
template <bool RES> constexpr int planes() { return RES ? 10 : 6; }
template <bool RES> constexpr int tile_words() { return planes<RES>() * MM_PLANE; }
constexpr int MM_PASS_MIN = 64;           // right-hand sides per pass, at least (mm_pass)
constexpr size_t MM_PASS_BYTES = size_t(4) << 30;   // operand tiles of a pass, above that many
constexpr int EXP_NONE = -200;            // exponent of a scale for zeros: below every other

__device__ __forceinline__ void mma16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
                 : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
                 : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
// the same with BF16 operands
__device__ __forceinline__ void mma16b(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2])
{
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
        : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}
__device__ __forceinline__ uint32_t h2(float a, float b)
{
    const __half2 v = __floats2half2_rn(a, b);
    return *reinterpret_cast<const uint32_t *>(&v);
}

// the planes of a pair of values (the smaller K in the lower half): each in three BF16 parts, rounded to nearest, exactly
__device__ __forceinline__ void split_pair(float a, float b, uint32_t (&p)[3])
{
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        asm("cvt.rn.bf16x2.f32 %0, %1, %2;" : "=r"(p[i]) : "f"(b), "f"(a));
        a = __fsub_rn(a, __uint_as_float(p[i] << 16));
        b = __fsub_rn(b, __uint_as_float(p[i] & 0xffff0000u));
    }
}

// The digit and sum steps run on packed pairs (k_dot2.cuh fma2, add2, sub2): two operations an
// issue slot, which is what bounds them beside the matrix instructions.
// the nearest integers of |v| < 2^22 (ties to even)
__device__ __forceinline__ float2 nearest(float2 v) { return sub2(add2(v, dup(12582912.f)), dup(12582912.f)); }
__device__ __forceinline__ float2 times(float2 v, float s) { return fma2(v, dup(s), dup(0.f)); }
// the planes of a pair of values v + lo, |v| <= 1, |lo| at most half an ulp of v: digits d1 .. d4 and the
// rest.  The trailing part joins where its bits begin, in the third digit.
__device__ __forceinline__ void split_pair(float2 v, float2 lo, uint32_t (&p)[5])
{
    auto put = [&](int i, float2 d) { p[i] = h2(d.x, d.y); };
    float2 t = times(v, 256.f), d = nearest(t);
    put(0, d);
    t = times(sub2(t, d), 512.f);
    d = nearest(t);
    put(1, d);
    t = times(sub2(t, d), 512.f);
    const float2 l = times(lo, 67108864.f);
    d = nearest(add2(t, l));
    put(2, d);
    t = times(add2(sub2(t, d), l), 512.f);
    d = nearest(t);
    put(3, d);
    put(4, times(sub2(t, d), 512.f));
}

__device__ __forceinline__ float pow2f(int e) { return __int_as_float((min(max(e, -126), 127) + 127) << 23); }
// v 2^e, in two factors so that every exponent a scale of FP32 data can have (below 252 either
// way) is taken whole: a factor cut off at the range of a float would be missing from the result
__device__ __forceinline__ float times_pow2(float v, int e)
{
    const int h = e / 2;
    return v * pow2f(h) * pow2f(e - h);
}
// 2^e over the whole range of a float, the subnormal powers too (0 below, infinite above)
__device__ __forceinline__ float pow2x(int e)
{
    if (e >= -126) return e > 127 ? __int_as_float(0x7f800000) : __int_as_float((e + 127) << 23);
    return e >= -149 ? __int_as_float(1 << (e + 149)) : 0.f;
}
// the least e with v <= 2^e (0 for 0 and for values that are not finite)
__device__ __forceinline__ int ceil_exp(float v)
{
    if (!(v > 0.f) || !isfinite(v)) return 0;
    int e;
    const float f = frexpf(v, &e);
    return f == 0.5f ? e - 1 : e;
}

// ---- x: scale per right-hand side, operand tiles --------------------------------

// ex[r] = the least e with |x_r|_inf <= 2^e; one CTA per right-hand side
// (245 KB of x at 30,720 unknowns: a few us beside products of milliseconds)
__global__ void __launch_bounds__(1024)
k_mm_max(const float2 *__restrict__ x, int64_t pN, int *__restrict__ ex)
{
    __shared__ float sm[32];
    const float4 *v = reinterpret_cast<const float4 *>(x + blockIdx.x * pN);   // pN is even
    float m = 0.f;
    for (int64_t i = threadIdx.x; i < pN / 2; i += 1024) {
        const float4 a = v[i];
        m = fmaxf(fmaxf(m, fmaxf(fabsf(a.x), fabsf(a.y))), fmaxf(fabsf(a.z), fabsf(a.w)));
    }
    m = warp_max(m);
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
        m = warp_max(sm[threadIdx.x]);
        if (threadIdx.x == 0) ex[blockIdx.x] = ceil_exp(m);
    }
}

// operand tiles of x: chunk of 16 unknowns (a warp each) x tile of 16 right-hand sides (blockIdx.y).
// ex: the product's scales (k_mm_max); the residual's own, of a chunk and right-hand side each, are
// formed here and written to ex[chunk * rp + r].
template <bool RES>
__global__ void __launch_bounds__(128)
k_mm_split(const XChunk *__restrict__ xch, int n_xch, const float2 *__restrict__ x, int64_t pN, int nrhs,
           int *__restrict__ ex, int rp, uint32_t *__restrict__ xt)
{
    const int ch = blockIdx.x * 4 + (threadIdx.x >> 5), lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    if (ch >= n_xch) return;
    const XChunk c = xch[ch];
    uint32_t *w = xt + ((int64_t)blockIdx.y * n_xch + ch) * tile_words<RES>() + t * 8 + g;
    float4 v[4];
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int q = blockIdx.y * 16 + g + 8 * (r & 1), k = 2 * t + 8 * (r >> 1);
        v[r] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (q < nrhs && k < c.len) {
            v[r] = *reinterpret_cast<const float4 *>(x + q * pN + c.off + k);
            if (k + 1 >= c.len) v[r].z = v[r].w = 0.f;
        }
    }
    int e[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {                  // right-hand sides g and g + 8
        const int q = blockIdx.y * 16 + g + 8 * h;
        if constexpr (RES) {
            float m = 0.f;
#pragma unroll
            for (int r = h; r < 4; r += 2)
                m = fmaxf(m, fmaxf(fmaxf(fabsf(v[r].x), fabsf(v[r].y)), fmaxf(fabsf(v[r].z), fabsf(v[r].w))));
            m = fmaxf(m, __shfl_xor_sync(FULL, m, 1));
            m = fmaxf(m, __shfl_xor_sync(FULL, m, 2));
            e[h] = m > 0.f ? ceil_exp(m) : EXP_NONE;
            if (t == 0) ex[(int64_t)ch * rp + q] = e[h];
        } else {
            e[h] = q < nrhs ? ex[q] : 0;
        }
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
        const int n = -e[r & 1];
        const float4 f = make_float4(times_pow2(v[r].x, n), times_pow2(v[r].y, n), times_pow2(v[r].z, n), times_pow2(v[r].w, n));
        constexpr int H = planes<RES>() / 2;
        uint32_t re[H], im[H];
        if constexpr (RES) {
            split_pair(make_float2(f.x, f.z), dup(0.f), re);
            split_pair(make_float2(f.y, f.w), dup(0.f), im);
        } else {
            split_pair(f.x, f.z, re);
            split_pair(f.y, f.w, im);
        }
#pragma unroll
        for (int p = 0; p < H; ++p) {
            w[p * MM_PLANE + r * 32] = re[p];
            w[(H + p) * MM_PLANE + r * 32] = im[p];
        }
    }
}

// the scales of T: ext[chunk * rp + r] = the largest of the x scales under the chunk's rank rows (tin:
// per T pair 4 * first x chunk + number of them - 1 of its input cluster, -1: none), so that with the
// W rows scaled to a 1-norm of 1 no T exceeds it
__global__ void __launch_bounds__(256)
k_mm_tscale(const int32_t *__restrict__ tin, int64_t n_tch, const int *__restrict__ ex, int rp, int *__restrict__ ext)
{
    const int64_t i = blockIdx.x * 256ll + threadIdx.x;
    if (i >= n_tch * rp) return;
    const int64_t c = i / rp;
    const int r = (int)(i - c * rp);
    int e = EXP_NONE, last = -1;
#pragma unroll
    for (int p = 0; p < MM_K / 2; ++p) {
        const int v = tin[c * (MM_K / 2) + p];
        if (v < 0 || v == last) continue;
        last = v;
        for (int q = 0; q <= (v & 3); ++q) e = max(e, ex[(int64_t)((v >> 2) + q) * rp + r]);
    }
    ext[i] = e;
}

// ---- operands of the blocks -------------------------------------------------------

// the B operands of one chunk and 8 outputs from the lane's four complex values (K 2t, 2t + 1,
// 2t + 8, 2t + 9 of output g): planes [part or digit][register]
template <bool RES> struct BFrag { uint32_t re[planes<RES>() / 2][2], im[planes<RES>() / 2][2]; };

// tile: an 8 x 16 tile of an operand stream in shared memory, two planes of 16 bytes a lane; scale (the
// residual's): what brings the lane's output row to at most 1
template <bool RES>
__device__ __forceinline__ void make_b(const unsigned char *tile, int lane, BFrag<RES> &b, float scale = 1.f)
{
    constexpr int H = planes<RES>() / 2;
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        const float4 v = *reinterpret_cast<const float4 *>(tile + q * 512 + lane * 16);
        uint32_t re[H], im[H];
        if constexpr (RES) {
            split_pair(times(make_float2(v.x, v.z), scale), dup(0.f), re);
            split_pair(times(make_float2(v.y, v.w), scale), dup(0.f), im);
        } else {
            split_pair(v.x, v.z, re);
            split_pair(v.y, v.w, im);
        }
#pragma unroll
        for (int p = 0; p < H; ++p) {
            b.re[p][q] = re[p];
            b.im[p][q] = im[p];
        }
    }
}
constexpr int MM_TILE = 1024;             // bytes of an 8 x 16 tile of a stream

__device__ __forceinline__ void negate(uint32_t (&n)[2], const uint32_t (&b)[2])
{
    n[0] = b[0] ^ 0x80008000u;
    n[1] = b[1] ^ 0x80008000u;
}

// plane p of an operand tile in shared memory (`tile`: the lane's word)
__device__ __forceinline__ void load_plane(uint32_t (&a)[4], const uint32_t *tile, int p)
{
#pragma unroll
    for (int r = 0; r < 4; ++r) a[r] = tile[p * MM_PLANE + r * 32];
}

// sums of one tile of 16 right-hand sides x 8 outputs
template <bool RES> struct Acc;
template <> struct Acc<false> {
    float s[2][4];              // re, im
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) s[0][i] = s[1][i] = 0.f;
    }
};
// one chunk into N tiles of 8 outputs (the products of the N tiles interleaved: a tile alone is
// two chains of dependent instructions): A operand planes at `tile` (the lane's word), B operands b.
// The small products first, so that only the last two instructions truncate at the sum's own size.
template <int N>
__device__ __forceinline__ void mm_chunk(Acc<false> (&s)[N], const uint32_t *tile, const BFrag<false> (&b)[N])
{
    float c[N][2][4] = {};
    uint32_t xr[4], xi[4];
    auto terms = [&](int q) {
#pragma unroll
        for (int n = 0; n < N; ++n) {
            mma16b(c[n][0], xr, b[n].re[q]);
            mma16b(c[n][1], xr, b[n].im[q]);
        }
#pragma unroll
        for (int n = 0; n < N; ++n) {
            uint32_t m[2];
            negate(m, b[n].im[q]);
            mma16b(c[n][0], xi, m);
            mma16b(c[n][1], xi, b[n].re[q]);
        }
    };
#pragma unroll
    for (int p = 2; p >= 0; --p) {                 // parts p of x with parts 2 - p .. 0 of the block
        load_plane(xr, tile, p);
        load_plane(xi, tile, 3 + p);
#pragma unroll
        for (int q = 2 - p; q >= 0; --q) terms(q);
    }
#pragma unroll
    for (int n = 0; n < N; ++n)
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            s[n].s[0][i] += c[n][0][i];
            s[n].s[1][i] += c[n][1][i];
        }
}
template <> struct Acc<true> {
    float2 hi[2][2], lo[2][2];      // re, im; right-hand sides g and g + 8; the pair of outputs
    __device__ __forceinline__ void zero()
    {
#pragma unroll
        for (int p = 0; p < 2; ++p)
#pragma unroll
            for (int i = 0; i < 2; ++i) hi[p][i] = lo[p][i] = dup(0.f);
    }
    // one chunk: digit p of x times digits 0 .. 4 - p of the block into h[p ..], then f times the weighted
    // sum (in units of 2^-16) into the running double-float.  h0 + 2^-9 h1 and that + 2^-18 h2 are
    // formed by the short form of TwoSum, exactly: where the second term is the larger one, it is at most
    // 2^13 (2^5), and the sum of two multiples of 2^-9 (2^-18) of that size is a float.
    __device__ __forceinline__ void chunk(const uint32_t *tile, const BFrag<true> &b, const float2 (&f)[2])
    {
        float h[5][2][4] = {};
#pragma unroll
        for (int p = 0; p < 5; ++p) {
            uint32_t xr[4], xi[4];
            load_plane(xr, tile, p);
            load_plane(xi, tile, 5 + p);
#pragma unroll
            for (int q = 0; q < 5 - p; ++q) {
                mma16(h[p + q][0], xr, b.re[q]);
                mma16(h[p + q][1], xr, b.im[q]);
            }
#pragma unroll
            for (int q = 0; q < 5 - p; ++q) {
                uint32_t n[2];
                negate(n, b.im[q]);
                mma16(h[p + q][0], xi, n);
                mma16(h[p + q][1], xi, b.re[q]);
            }
        }
#pragma unroll
        for (int c = 0; c < 2; ++c)
#pragma unroll
            for (int i = 0; i < 2; ++i) {
                float2 w[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) w[q] = make_float2(h[q][c][2 * i], h[q][c][2 * i + 1]);
                const float2 s = fma2(w[1], dup(0x1p-9f), w[0]);
                const float2 e = fma2(w[1], dup(0x1p-9f), sub2(w[0], s));
                const float2 v = fma2(w[2], dup(0x1p-18f), s);
                const float2 e2 = fma2(w[2], dup(0x1p-18f), sub2(s, v));
                const float2 l = fma2(w[4], dup(0x1p-36f), fma2(w[3], dup(0x1p-27f), add2(e, e2)));
                const float2 vf = fma2(v, f[i], dup(0.f));
                const float2 a = hi[c][i], n = add2(a, vf), bb = sub2(n, a);
                const float2 e3 = add2(sub2(a, sub2(n, bb)), sub2(vf, bb));
                hi[c][i] = n;
                lo[c][i] = add2(lo[c][i], fma2(l, f[i], e3));
            }
    }
};

// ---- copies ------------------------------------------------------------------------

__device__ __forceinline__ uint32_t su32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp16(uint32_t dst, const void *src)
{
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
// waits until at most N of this thread's latest groups are in flight
template <int N> __device__ __forceinline__ void cp_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// ---- stage 1: T = W X --------------------------------------------------------------

// per warp: two halves of four W tiles and (the residual) their rows' exponents
template <bool RES> constexpr int s1_half() { return 4 * (MM_TILE + (RES ? 32 : 0)); }
template <bool RES, int MT> constexpr int s1_smem() { return 4 * MT * tile_words<RES>() * 4 + MMW * 2 * s1_half<RES>(); }

struct MmS1Args {
    const MmBatch *batches;
    const int32_t *tdst;
    const unsigned char *ws;  // operand stream
    const int *wrow;          // the residual: per stream tile its 8 rows' exponents
    const uint32_t *xt;
    uint32_t *tt;
    const int *ex, *ext;      // the residual: scales of x and of T, [chunk][rp]
    int64_t n_tch;
    int n_xch, n_tiles, groups, rp;
};

// One batch of W row tiles over an input cluster (blockIdx.x / groups) and MT tiles of 16
// right-hand sides (blockIdx.x % groups: the CTAs that read the same blocks run together, from L2): the cluster's x tiles are copied to shared memory once, each warp takes
// every 8th tile of 8 rows, the next one in flight while one is multiplied.
template <bool RES, int MT>
__global__ void __launch_bounds__(MMW * 32, 2)
k_mm_stage1(const MmS1Args A)
{
    extern __shared__ __align__(128) unsigned char sm1[];
    constexpr int TW = tile_words<RES>(), HALF = s1_half<RES>();
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const MmBatch B = A.batches[blockIdx.x / A.groups];
    const int nch = (B.klen + MM_K - 1) / MM_K;
    const int m0 = blockIdx.x % A.groups * MT;
    uint32_t *xs = reinterpret_cast<uint32_t *>(sm1);
    unsigned char *wr = sm1 + 4 * MT * TW * 4 + w * 2 * HALF;
    auto fetch = [&](int it, int h) {
        const int64_t pos = (int64_t)B.pos + (int64_t)it * nch;
        const unsigned char *src = A.ws + pos * MM_TILE + lane * 16;
        const uint32_t d = su32(wr + h * HALF + lane * 16);
        for (int c = 0; c < 2 * nch; ++c) cp16(d + c * 512, src + c * 512);
        if constexpr (RES) {
            if (lane < 2 * nch) cp16(d + 4 * MM_TILE, A.wrow + pos * 8 + lane * 4);
        }
    };
    for (int i = threadIdx.x; i < nch * MT * (TW / 4); i += MMW * 32) {
        const int c = i / (MT * (TW / 4)), m = i / (TW / 4) % MT, o = i % (TW / 4);
        if (m0 + m < A.n_tiles)
            cp16(su32(xs + (c * MT + m) * TW + 4 * o), A.xt + ((int64_t)(m0 + m) * A.n_xch + B.xg0 + c) * TW + 4 * o);
    }
    if (w < B.ntiles) fetch(w, 0);
    cp_commit();
    int ex[4][2] = {};                             // of right-hand sides g and g + 8
    if constexpr (RES) {
        static_assert(!RES || MT == 1, "one tile of right-hand sides a lane's scales");
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (c < nch) {
                const int *e = A.ex + (int64_t)(B.xg0 + c) * A.rp + 16 * m0 + g;
                ex[c][0] = e[0];
                ex[c][1] = e[8];
            }
    }
    cp_wait<0>();
    __syncthreads();
    const uint32_t *xw = xs + t * 8 + g;
    int h = 0;
    for (int it = w; it < B.ntiles; it += MMW, h ^= 1) {
        const int dst = A.tdst[4 * (B.tile0 + it) + t];
        int eT[2] = {0, 0};                        // T's scales: its row pair belongs to this lane
        if constexpr (RES) {
            if (dst >= 0) {
                const int *e = A.ext + (int64_t)(dst >> 3) * A.rp + 16 * m0 + g;
                eT[0] = e[0];
                eT[1] = e[8];
            }
        }
        __syncwarp();                              // every lane is done with the half the next copy fills
        if (it + MMW < B.ntiles) fetch(it + MMW, h ^ 1);
        cp_commit();
        cp_wait<1>();
        __syncwarp();                              // the warp's copies of this tile have landed
        Acc<RES> acc[MT][1];
#pragma unroll
        for (int m = 0; m < MT; ++m) acc[m][0].zero();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
            if (c >= nch) break;
            BFrag<RES> f[1];
            if constexpr (RES) {
                const int ew = reinterpret_cast<const int *>(wr + h * HALF + 4 * MM_TILE)[8 * c + g];
                make_b<RES>(wr + h * HALF + c * MM_TILE, lane, f[0], pow2f(-ew));
                const int w0 = __shfl_sync(FULL, ew, 8 * t), w1 = __shfl_sync(FULL, ew, 8 * t + 4);
                const float2 sc[2] = {make_float2(pow2x(w0 + ex[c][0] - eT[0] - 16), pow2x(w1 + ex[c][0] - eT[0] - 16)),
                                      make_float2(pow2x(w0 + ex[c][1] - eT[1] - 16), pow2x(w1 + ex[c][1] - eT[1] - 16))};
                acc[0][0].chunk(xw + c * TW, f[0], sc);
            } else {
                make_b<RES>(wr + h * HALF + c * MM_TILE, lane, f[0]);
#pragma unroll
                for (int m = 0; m < MT; ++m) mm_chunk<1>(acc[m], xw + (c * MT + m) * TW, f);
            }
        }
        if (dst < 0) continue;
        // accumulators 0, 1 (right-hand side g) and 2, 3 (g + 8) are the K pair dst of T
        const int pr = dst & 7;
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            if (m0 + m >= A.n_tiles) break;
            uint32_t *o = A.tt + ((int64_t)(m0 + m) * A.n_tch + (dst >> 3)) * TW + (pr >> 2) * 64 + (pr & 3) * 8 + g;
#pragma unroll
            for (int q = 0; q < 2; ++q)
#pragma unroll
                for (int c = 0; c < 2; ++c) {   // re, im
                    constexpr int H = planes<RES>() / 2;
                    uint32_t p[H];
                    if constexpr (RES) {
                        float2 v, l;
                        two_sum(acc[m][0].hi[c][q].x, acc[m][0].lo[c][q].x, v.x, l.x);
                        two_sum(acc[m][0].hi[c][q].y, acc[m][0].lo[c][q].y, v.y, l.y);
                        split_pair(v, l, p);
                    } else {
                        split_pair(acc[m][0].s[c][2 * q], acc[m][0].s[c][2 * q + 1], p);
                    }
#pragma unroll
                    for (int j = 0; j < H; ++j) __stcs(o + (H * c + j) * MM_PLANE + q * 32, p[j]);
                }
        }
    }
}

// ---- output stage ------------------------------------------------------------------

struct MmOutArgs {
    const MmUnit *units;
    const int32_t *ca;       // per chunk: its split-x chunk, or -1 - its T chunk
    const int *eout;         // per output cluster: E
    const unsigned char *os; // operand stream
    const uint32_t *xt, *tt;
    int n_xch, n_tiles, nrhs;
    int64_t n_tch;
    const int *ex, *ext;     // exponents of the scales: the product's per right-hand side (k_mm_max); the residual's
                             // of x and of T, [chunk][rp]
    const int *orow;         // the residual: per stream tile its 8 rows' exponents
    int rp;
    int groups;              // CTAs of a unit, over the right-hand sides
};

// The copies of a K group: T threads that work on the same chunks, each chunk's stream tiles and
// the operand tiles of `mtiles` tiles of right-hand sides in one of the stages of the group's
// shared memory.  The operand tile index of the next chunk is loaded one chunk ahead.
template <bool RES> struct Pipe {
    static constexpr int NB = RES ? 2 : 4;        // 16-byte pieces of a chunk's stream per thread, at most
    static constexpr int TW = tile_words<RES>();
    uint32_t base;
    const unsigned char *smem, *src;               // src: the thread's piece of the chunk to copy next
    const int *rows;                               // the residual: the piece of its rows' exponents
    int gt, T, tiles, mtiles, m0, n_tiles, stages, bsz, ssz, a, step;
    __device__ __forceinline__ void init(const MmOutArgs &A, const MmUnit &U, unsigned char *region, int bytes, int gt_, int T_,
                                         int room, int mt, int m0_, int kw, int ks)
    {
        base = su32(region);
        smem = region;
        gt = gt_; T = T_; mtiles = mt; m0 = m0_; n_tiles = A.n_tiles;
        tiles = (U.mlen + 7) / 8;
        bsz = room * (MM_TILE + (RES ? 32 : 0));
        ssz = bsz + mtiles * TW * 4 + (RES ? 64 : 0);
        stages = min(6, bytes / ssz);
        step = ks * tiles * MM_TILE;
        src = A.os + ((int64_t)U.pos + kw * tiles) * MM_TILE + gt * 16;
        if constexpr (RES) rows = A.orow + ((int64_t)U.pos + kw * tiles) * 8 + gt * 4;
    }
    __device__ __forceinline__ void copy(const MmOutArgs &A, int stage)
    {
        const uint32_t st = base + stage * ssz;
#pragma unroll
        for (int j = 0; j < NB; ++j)
            if (gt + T * j < tiles * (MM_TILE / 16)) cp16(st + (gt + T * j) * 16, src + T * j * 16);
        src += step;
        const uint32_t *tl = a < 0 ? A.tt + (int64_t)(-1 - a) * TW : A.xt + (int64_t)a * TW;
        const int64_t stride = (a < 0 ? A.n_tch : A.n_xch) * TW;
        for (int q = gt; q < mtiles * (TW / 4); q += T) {
            const int m = q / (TW / 4), o = q % (TW / 4);
            if (m0 + m < n_tiles) cp16(st + bsz + q * 16, tl + (m0 + m) * stride + 4 * o);
        }
        if constexpr (RES) {                       // T >= 32 > 2 tiles + 4: two pieces by different threads
            if (gt < 2 * tiles) cp16(st + (bsz - tiles * 32) + gt * 16, rows);
            rows += step / (MM_TILE / 8);
            const int q = gt - (T - 4);
            if (q >= 0) cp16(st + bsz + TW * 4 + q * 16, (a < 0 ? A.ext + (int64_t)(-1 - a) * A.rp : A.ex + (int64_t)a * A.rp) + 16 * m0 + 4 * q);
        }
    }
    // the residual: exponents of output tile n's rows, and of the chunk's operand for the 16 right-hand sides
    __device__ __forceinline__ const int *row_exp(int stage, int n) const
    {
        return reinterpret_cast<const int *>(smem + stage * ssz + bsz - tiles * 32) + 8 * n;
    }
    __device__ __forceinline__ const int *operand_exp(int stage) const
    {
        return reinterpret_cast<const int *>(smem + stage * ssz + bsz + TW * 4);
    }
    __device__ __forceinline__ const uint32_t *tile(int stage, int m) const
    {
        return reinterpret_cast<const uint32_t *>(smem + stage * ssz + bsz) + m * TW;
    }
    __device__ __forceinline__ const unsigned char *values(int stage, int n) const { return smem + stage * ssz + n * MM_TILE; }
    // the pipeline over chunks c0, c0 + ks, ... < c1: body(stage) for each; the group's threads meet at
    // the named barrier `bar` once a chunk
    template <class Body>
    __device__ __forceinline__ void run(const MmOutArgs &A, int c0, int c1, int ks, int bar, Body body)
    {
        if (stages >= 5) run_stages<5>(A, c0, c1, ks, bar, body);
        else if (stages >= 3) run_stages<3>(A, c0, c1, ks, bar, body);
        else run_stages<2>(A, c0, c1, ks, bar, body);
    }
    template <int S, class Body>
    __device__ __forceinline__ void run_stages(const MmOutArgs &A, int c0, int c1, int ks, int bar, Body body)
    {
        const int n = c0 < c1 ? (c1 - c0 + ks - 1) / ks : 0;
        const int32_t *ca = A.ca + c0;
        if (n > 0) a = *ca;
#pragma unroll
        for (int q = 0; q < S - 1; ++q) {
            if (q < n) copy(A, q);
            cp_commit();
            ca += ks;
            if (q + 1 < n) a = *ca;
        }
        int st = 0, nx = S - 1;                    // the stage of chunk q, and of chunk q + S - 1
        for (int q = 0; q < n; ++q) {
            cp_wait<S - 2>();
            asm volatile("bar.sync %0, %1;" ::"r"(bar), "r"(T) : "memory");
            if (q + S - 1 < n) copy(A, nx);
            cp_commit();
            ca += ks;
            if (q + S < n) a = *ca;
            body(st);
            st = st + 1 == S ? 0 : st + 1;
            nx = nx + 1 == S ? 0 : nx + 1;
        }
        cp_wait<0>();
    }
};

constexpr int MM_SMEM = 112 * 1024;               // two CTAs an SM

// Product: one unit (blockIdx.x / groups) for MT x mw tiles of 16 right-hand sides.  The 8
// warps: 16 outputs each (the fastest index), mw groups of MT right-hand-side tiles, and what
// is left of them along K, as far as two stages of their copies fit; every warp adds its sums into
// z (vector atomics).
template <int MT>
__global__ void __launch_bounds__(MMW * 32, 2)
k_mm_out(MmOutArgs p, int mw, float2 *__restrict__ z, int64_t pN)
{
    extern __shared__ __align__(128) unsigned char smo[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const MmUnit U = p.units[blockIdx.x / p.groups];
    const int nt = (U.mlen + 15) / 16, gw = nt * mw, kw = w / gw, wi = w - kw * gw;
    const int ks = min(MMW / gw, MM_SMEM / (2 * (2 * nt * MM_TILE + MT * mw * tile_words<false>() * 4)));
    if (kw >= ks) return;
    const int n0 = 16 * (wi % nt), mi = (wi / nt) * MT, mb = (int)(blockIdx.x % p.groups) * mw * MT, m0 = mb + mi;
    const int E = p.eout[U.cl];
    Acc<false> acc[MT][2];
#pragma unroll
    for (int m = 0; m < MT; ++m) { acc[m][0].zero(); acc[m][1].zero(); }
    Pipe<false> P;
    const int region = MM_SMEM / ks / 128 * 128;
    P.init(p, U, smo + kw * region, region, wi * 32 + lane, gw * 32, 2 * nt, MT * mw, mb, kw, ks);
    P.run(p, U.c0 + kw, U.c1, ks, 1 + kw, [&](int st) {
        BFrag<false> f[2];
#pragma unroll
        for (int n = 0; n < 2; ++n) make_b<false>(P.values(st, n0 / 8 + n), lane, f[n]);
#pragma unroll
        for (int m = 0; m < MT; ++m) {
            if (m0 + m >= p.n_tiles) break;
            const uint32_t *tile = P.tile(st, mi + m) + t * 8 + g;
            mm_chunk<2>(acc[m], tile, f);
        }
    });
#pragma unroll
    for (int m = 0; m < MT; ++m)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int r = 16 * (m0 + m) + g + 8 * h;
            if (r >= p.nrhs) continue;
            const int e = p.ex[r] - E;
#pragma unroll
            for (int n = 0; n < 2; ++n) {
                const int i = n0 + 8 * n + 2 * t;
                const float2 a = make_float2(times_pow2(acc[m][n].s[0][2 * h], e), times_pow2(acc[m][n].s[1][2 * h], e));
                const float2 b = make_float2(times_pow2(acc[m][n].s[0][2 * h + 1], e), times_pow2(acc[m][n].s[1][2 * h + 1], e));
                float2 *zz = z + (int64_t)r * pN + U.out0 + i;
                if (i + 1 < U.mlen) red2(zz, a, b);
                else if (i < U.mlen) red1(zz, a);
            }
        }
}

// FP64-class residual products: one unit (blockIdx.x / groups) for a tile of 16 right-hand
// sides.  The 8 warps: 8 outputs each, the rest along K; the K groups' double-float
// sums are added in a fixed order, the unit's sums stored once in FP64: no atomics, the
// result does not depend on scheduling.
__global__ void __launch_bounds__(MMW * 32, 2)
k_mm_resid(MmOutArgs p, double2 *__restrict__ own, int64_t pstride, int64_t pN)
{
    extern __shared__ __align__(128) unsigned char smo[];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
    const MmUnit U = p.units[blockIdx.x / p.groups];
    const int nt = (U.mlen + 7) / 8, ks = MMW / nt, kw = w / nt, wi = w - kw * nt, m0 = (int)(blockIdx.x % p.groups);
    const int n0 = 8 * wi;
    const int E = p.eout[U.cl];
    Acc<true> acc;
    acc.zero();
    if (kw < ks) {
        Pipe<true> P;
        const int region = MM_SMEM / ks / 128 * 128;
        P.init(p, U, smo + kw * region, region, wi * 32 + lane, nt * 32, nt, 1, m0, kw, ks);
        P.run(p, U.c0 + kw, U.c1, ks, 1 + kw, [&](int st) {
            BFrag<true> f;
            const int eb = P.row_exp(st, wi)[g];
            make_b<true>(P.values(st, wi), lane, f, pow2f(-eb));
            const int *ea = P.operand_exp(st) + g;
            const int b0 = __shfl_sync(FULL, eb, 8 * t) - E - 16, b1 = __shfl_sync(FULL, eb, 8 * t + 4) - E - 16;
            const float2 sc[2] = {make_float2(pow2x(ea[0] + b0), pow2x(ea[0] + b1)),
                                  make_float2(pow2x(ea[8] + b0), pow2x(ea[8] + b1))};
            acc.chunk(P.tile(st, 0) + t * 8 + g, f, sc);
        });
    }
    float *hi = reinterpret_cast<float *>(acc.hi), *lo = reinterpret_cast<float *>(acc.lo);   // 4 (re, im) + 2 h + j
    if (ks > 1) {
        float(*sm)[16][32] = reinterpret_cast<float(*)[16][32]>(smo);
        __syncthreads();                            // every group is done with its stages
#pragma unroll
        for (int i = 0; i < 8; ++i) {
            sm[w][2 * i][lane] = hi[i];
            sm[w][2 * i + 1][lane] = lo[i];
        }
        __syncthreads();
        if (kw == 0)
            for (int q = 1; q < ks; ++q)
#pragma unroll
                for (int i = 0; i < 8; ++i) {
                    const df v = df_add(df{hi[i], lo[i]}, df{sm[w + q * nt][2 * i][lane], sm[w + q * nt][2 * i + 1][lane]});
                    hi[i] = v.hi;
                    lo[i] = v.lo;
                }
    }
    if (kw != 0) return;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
        const int r = 16 * m0 + g + 8 * h;
        if (r >= p.nrhs) continue;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
            const int i = n0 + 2 * t + j, a = 2 * h + j;
            if (i < U.mlen)
                own[(int64_t)U.part * pstride + (int64_t)r * pN + U.out0 + i] =
                    make_double2((double)hi[a] + (double)lo[a], (double)hi[4 + a] + (double)lo[4 + a]);
        }
    }
}

// ---- scales, once per operator -------------------------------------------------------

// Per directed product (a warp each): low-rank, et of every W row from its 1-norm (FP32, rounded
// up, of the row scaled to 1 so that it cannot overflow) into wexp and, negated, into rexp, and
// E's bound et - exponent(max Y row); dense, E's bound from the block's largest component.  A
// row pair whose W row is zero gives nothing: its Y row is packed as zeros (ROW_OFF).
constexpr int ROW_OFF = -(1 << 20);
__global__ void __launch_bounds__(256)
k_mm_prep(const MmSet *__restrict__ sets, int64_t n, const float2 *__restrict__ pool, int *__restrict__ wexp,
          int *__restrict__ rexp, int *__restrict__ eout)
{
    const int lane = threadIdx.x & 31;
    const int64_t nw = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t q = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); q < n; q += nw) {
        const MmSet S = sets[q];
        int bound = 1000;
        if (S.rank == 0) {
            float m = 0.f;
            for (int i = 0; i < S.y_ld; ++i)
                for (int j = lane; j < S.wlen; j += 32) m = fmaxf(m, linf(pool[S.w + (int64_t)i * S.w_ld + j]));
            m = warp_max(m);
            if (m > 0.f) bound = -ceil_exp(m);
        }
        for (int l = 0; l < S.rank; ++l) {
            float w = 0.f, a = 0.f, m = 0.f;
            for (int j = lane; j < S.wlen; j += 32) w = fmaxf(w, linf(pool[S.w + (int64_t)l * S.w_ld + j]));
            for (int i = lane; i < S.ylen; i += 32) m = fmaxf(m, linf(pool[S.y + (int64_t)l * S.y_ld + i]));
            w = warp_max(w);
            m = warp_max(m);
            const int ew = -ceil_exp(w);
            for (int j = lane; j < S.wlen; j += 32) {
                const float2 v = pool[S.w + (int64_t)l * S.w_ld + j];
                a = __fadd_ru(a, __fadd_ru(fabsf(times_pow2(v.x, ew)), fabsf(times_pow2(v.y, ew))));
            }
#pragma unroll
            for (int s = 16; s >= 1; s >>= 1) a = __fadd_ru(a, __shfl_xor_sync(FULL, a, s));
            const int et = ew - ceil_exp(a);
            if (lane == 0) {
                wexp[2 * (int64_t)S.p0 + l] = et;
                rexp[2 * (int64_t)S.t0 + l] = w == 0.f ? ROW_OFF : -et;
            }
            if (m > 0.f && w != 0.f) bound = min(bound, et - ceil_exp(m));
        }
        if (lane == 0 && bound < 1000) atomicMin(eout + S.cl, bound);
    }
}
// rexp = E - et of every T row; clusters with nothing but zeros get E = 0
__global__ void __launch_bounds__(256)
k_mm_rexp(const MmSet *__restrict__ sets, int64_t n, int *__restrict__ rexp, const int *__restrict__ eout)
{
    for (int64_t q = blockIdx.x * 256ll + threadIdx.x; q < n; q += gridDim.x * 256ll) {
        const MmSet S = sets[q];
        for (int l = 0; l < S.rank; ++l) {
            int &v = rexp[2 * (int64_t)S.t0 + l];
            if (v != ROW_OFF) v += eout[S.cl];
        }
    }
}
__global__ void k_mm_eout(int *eout, int n, int set)
{
    const int i = blockIdx.x * 256 + threadIdx.x;
    if (i < n && (set || eout[i] == 1000)) eout[i] = set ? 1000 : 0;
}

// ---- operand streams, once per operator ---------------------------------------------

// the lane's four values times 2^e, and the exponent of the tile's row (the residual's scale; not below
// -120, so that its inverse is a float)
__device__ __forceinline__ void pack_tile(float4 *dst, int *row, const float2 (&v)[4], const int (&e)[4], int lane)
{
    float f[8];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        f[2 * q] = ldexpf(v[q].x, e[q]);
        f[2 * q + 1] = ldexpf(v[q].y, e[q]);
    }
    dst[lane] = make_float4(f[0], f[1], f[2], f[3]);
    dst[32 + lane] = make_float4(f[4], f[5], f[6], f[7]);
    float m = 0.f;
#pragma unroll
    for (int q = 0; q < 8; ++q) m = fmaxf(m, fabsf(f[q]));
    m = fmaxf(m, __shfl_xor_sync(FULL, m, 1));
    m = fmaxf(m, __shfl_xor_sync(FULL, m, 2));
    if ((lane & 3) == 0) row[lane >> 2] = m > 0.f ? max(ceil_exp(m), -120) : -120;
}

// the output stream, a warp per chunk
__global__ void __launch_bounds__(256)
k_mm_pack_out(const MmChunk *__restrict__ chunks, int64_t n, const int64_t *__restrict__ rows, const int *__restrict__ rexp,
              const int *__restrict__ eout, const float2 *__restrict__ pool, unsigned char *__restrict__ os,
              int *__restrict__ orow, int32_t *__restrict__ ca)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    for (int64_t c = blockIdx.x * 8ll + (threadIdx.x >> 5); c < n; c += gridDim.x * 8ll) {
        const MmChunk C = chunks[c];
        if (lane == 0) ca[c] = C.kind == 2 ? -1 - C.a : C.a;
        int64_t off[4];
        int e[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const int k = 2 * t + (q & 1) + 8 * (q >> 1);
            off[q] = C.kind == 2 ? rows[C.src + k] : k < C.klen ? C.src + (C.kind == 0 ? k : (int64_t)k * C.ld) : -1;
            e[q] = C.kind == 2 ? rexp[C.src + k] : eout[C.cl];
        }
        for (int tl = 0; tl < C.tiles; ++tl) {
            const int i = 8 * tl + g;
            float2 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q)
                v[q] = off[q] >= 0 && i < C.olen ? pool[off[q] + (C.kind == 0 ? (int64_t)i * C.ld : i)] : make_float2(0.f, 0.f);
            pack_tile(reinterpret_cast<float4 *>(os + ((int64_t)C.pos + tl) * MM_TILE), orow + ((int64_t)C.pos + tl) * 8, v, e, lane);
        }
    }
}

// the stage-1 stream, a CTA per batch, a warp per tile of 8 W rows
__global__ void __launch_bounds__(256)
k_mm_pack_w(const MmBatch *__restrict__ batches, const MmPair *__restrict__ pairs, const int *__restrict__ wexp,
            const float2 *__restrict__ pool, unsigned char *__restrict__ ws, int *__restrict__ wrow, int32_t *__restrict__ tdst,
            int32_t *__restrict__ tin)
{
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    const MmBatch B = batches[blockIdx.x];
    const int nch = (B.klen + MM_K - 1) / MM_K;
    for (int it = threadIdx.x >> 5; it < B.ntiles; it += 8) {
        const int tile = B.tile0 + it;
        const MmPair P = pairs[4 * tile + (g >> 1)];
        const int64_t off = P.w < 0 || ((g & 1) && P.ld == 0) ? -1 : P.w + (g & 1) * (int64_t)P.ld;
        const int ew = wexp[8 * tile + g], e[4] = {ew, ew, ew, ew};
        if (lane < 4) {
            const MmPair Q = pairs[4 * tile + lane];
            tdst[4 * tile + lane] = Q.dst;
            if (Q.dst >= 0) tin[Q.dst] = Q.w < 0 ? -1 : 4 * B.xg0 + nch - 1;
        }
        for (int c = 0; c < nch; ++c) {
            float2 v[4];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                const int k = c * MM_K + 2 * t + (q & 1) + 8 * (q >> 1);
                v[q] = off >= 0 && k < B.klen ? pool[off + k] : make_float2(0.f, 0.f);
            }
            const int64_t pos = (int64_t)B.pos + (int64_t)it * nch + c;
            pack_tile(reinterpret_cast<float4 *>(ws + pos * MM_TILE), wrow + pos * 8, v, e, lane);
        }
    }
}

} // namespace

// scales and operand streams of a level's lists (device copies M; wexp, rexp zeroed by the caller)
void launch_mm_pack(const LevelList &L, const MmPackArgs &M, const float2 *pool, cudaStream_t s)
{
    const int n_cl = M.n_cl;
    if (M.n_sets <= 0 || n_cl <= 0) return;
    k_mm_eout<<<(n_cl + 255) / 256, 256, 0, s>>>(L.d_mm_eout, n_cl, 1);
    k_mm_prep<<<(unsigned)std::min<int64_t>((M.n_sets + 7) / 8, 152 * 16), 256, 0, s>>>(M.sets, M.n_sets, pool, M.wexp, M.rexp,
                                                                                      L.d_mm_eout);
    k_mm_eout<<<(n_cl + 255) / 256, 256, 0, s>>>(L.d_mm_eout, n_cl, 0);
    k_mm_rexp<<<(unsigned)std::min<int64_t>((M.n_sets + 255) / 256, 4096), 256, 0, s>>>(M.sets, M.n_sets, M.rexp, L.d_mm_eout);
    k_mm_pack_out<<<(unsigned)std::min<int64_t>((M.n_chunks + 7) / 8, 152 * 32), 256, 0, s>>>(
        M.chunks, M.n_chunks, M.rows, M.rexp, L.d_mm_eout, pool, L.d_mm_os, L.d_mm_orow, L.d_mm_ca);
    if (L.mm_n_batch > 0)
        k_mm_pack_w<<<(unsigned)L.mm_n_batch, 256, 0, s>>>(L.d_mm_batch, M.pairs, M.wexp, pool, L.d_mm_ws, L.d_mm_wrow, L.d_mm_tdst, L.d_mm_tin);
}
size_t mm_stream_bytes(int64_t tiles) { return (size_t)tiles * MM_TILE; }

// right-hand sides per pass: all of them while x and T in operand layout fit MM_PASS_BYTES (a
// pass streams the blocks from HBM once), else whole groups of 64 that do
static int mm_pass(const LevelList &L, int nrhs, bool res)
{
    const size_t words = res ? tile_words<true>() : tile_words<false>();
    const size_t tile = words * sizeof(uint32_t) * ((size_t)L.mm_n_xch + (size_t)L.mm_n_tch);
    const int64_t fit = (int64_t)(MM_PASS_BYTES / std::max<size_t>(tile, 1)) * 16 / MM_PASS_MIN * MM_PASS_MIN;
    return (int)std::min<int64_t>(nrhs, std::max<int64_t>(fit, MM_PASS_MIN));
}

// bytes of the operand tiles (x, then T, then the scales' exponents) of a pass over nrhs
size_t mm_ws_bytes(const LevelList &L, int nrhs, bool res)
{
    const int pass = mm_pass(L, nrhs, res);
    const size_t tiles = (size_t)(pass + 15) / 16;
    const size_t words = res ? tile_words<true>() : tile_words<false>();
    const size_t chunks = (size_t)L.mm_n_xch + (size_t)L.mm_n_tch;
    return tiles * words * sizeof(uint32_t) * chunks + sizeof(int) * (res ? 16 * tiles * chunks : (size_t)pass);
}

namespace {
// shared memory of a kernel beyond the default, two CTAs an SM
void mm_attr(const void *kern, int smem)
{
    cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    cudaFuncSetAttribute(kern, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
}

// x of a pass into operand tiles, then stage 1
template <bool RES>
int mm_inputs(hm_matrix h, const LevelList &L, const float2 *x, int nr, uint32_t *xt, uint32_t *tt, int *ex, cudaStream_t s)
{
    const int tiles = (nr + 15) / 16, rp = 16 * tiles;
    int n = 1;
    if (!RES) {
        k_mm_max<<<nr, 1024, 0, s>>>(x, h->pN, ex);
        ++n;
    }
    k_mm_split<RES><<<dim3((unsigned)((L.mm_n_xch + 3) / 4), (unsigned)tiles), 128, 0, s>>>(L.d_mm_xch, (int)L.mm_n_xch, x,
                                                                                           h->pN, nr, ex, rp, xt);
    if (L.mm_n_batch == 0) return n;
    int *ext = ex + L.mm_n_xch * rp;
    if (RES) {
        k_mm_tscale<<<(unsigned)((L.mm_n_tch * rp + 255) / 256), 256, 0, s>>>(L.d_mm_tin, L.mm_n_tch, ex, rp, ext);
        ++n;
    }
    auto go = [&](auto kern, int mt, int smem) {
        mm_attr((const void *)kern, smem);
        const int groups = (tiles + mt - 1) / mt;
        const MmS1Args a{L.d_mm_batch, L.d_mm_tdst, L.d_mm_ws, L.d_mm_wrow, xt, tt, ex, RES ? ext : nullptr, L.mm_n_tch,
                         (int)L.mm_n_xch, tiles, groups, rp};
        kern<<<(unsigned)(groups * L.mm_n_batch), MMW * 32, smem, s>>>(a);
        ++n;
    };
    if constexpr (!RES) {
        if (tiles > 1) {
            go(k_mm_stage1<RES, 2>, 2, s1_smem<RES, 2>());
            return n;
        }
    }
    go(k_mm_stage1<RES, 1>, 1, s1_smem<RES, 1>());
    return n;
}
} // namespace

// z += M_level x for the level's small items and all right-hand sides; ws as mm_ws_bytes
int launch_mm_product(hm_matrix h, const LevelList &L, const float2 *x, float2 *z, int nrhs, void *ws, cudaStream_t s)
{
    if (L.mm_n_unit == 0 || nrhs <= 0) return 0;
    int n = 0;
    const int pass = mm_pass(L, nrhs, false);
    const size_t tiles_max = (size_t)(pass + 15) / 16;
    uint32_t *xt = (uint32_t *)ws, *tt = xt + tiles_max * tile_words<false>() * L.mm_n_xch;
    int *ex = (int *)(tt + tiles_max * tile_words<false>() * L.mm_n_tch);
    for (int r0 = 0; r0 < nrhs; r0 += pass) {
        const int nr = std::min(pass, nrhs - r0), tiles = (nr + 15) / 16;
        const float2 *xp = x + (int64_t)r0 * h->pN;
        n += mm_inputs<false>(h, L, xp, nr, xt, tt, ex, s) + 1;
        // tiles of 16 right-hand sides a warp up to 16 of them, 32 above, two such groups a CTA above 32
        const int mw = tiles > 2 ? 2 : 1, mt = tiles > 1 ? 2 : 1, groups = (tiles + mt * mw - 1) / (mt * mw);
        // the coarse units, with fewer sums to add into z, where they alone are four CTAs an SM
        const bool coarse = tiles > 2 && (int64_t)groups * L.mm_n_unit2 >= 4ll * h->num_sms;
        MmOutArgs a{coarse ? L.d_mm_unit2 : L.d_mm_unit, L.d_mm_ca, L.d_mm_eout, L.d_mm_os, xt, tt, (int)L.mm_n_xch,
                    tiles, nr, L.mm_n_tch, ex, nullptr, nullptr, 16 * tiles, groups};
        float2 *zp = z + (int64_t)r0 * h->pN;
        const unsigned units = (unsigned)(coarse ? L.mm_n_unit2 : L.mm_n_unit);
        auto go = [&](auto kern) {
            mm_attr((const void *)kern, MM_SMEM);
            kern<<<units * (unsigned)groups, MMW * 32, MM_SMEM, s>>>(a, mw, zp, h->pN);
        };
        if (mt == 1) go(k_mm_out<1>);
        else go(k_mm_out<2>);
    }
    return n;
}

// own[part][r][p] = the FP64-class sums of the level's small items' products, by part of the
// output cluster's units (rows no unit covers are left as they are)
int launch_mm_resid(hm_matrix h, const LevelList &L, const float2 *x, double2 *own, int64_t pstride, int nrhs, void *ws,
                    cudaStream_t s)
{
    if (L.mm_n_runit == 0 || nrhs <= 0) return 0;
    int n = 0;
    const int pass = mm_pass(L, nrhs, true);
    const size_t tiles_max = (size_t)(pass + 15) / 16;
    uint32_t *xt = (uint32_t *)ws, *tt = xt + tiles_max * tile_words<true>() * L.mm_n_xch;
    int *ex = (int *)(tt + tiles_max * tile_words<true>() * L.mm_n_tch);
    for (int r0 = 0; r0 < nrhs; r0 += pass) {
        const int nr = std::min(pass, nrhs - r0), tiles = (nr + 15) / 16;
        n += mm_inputs<true>(h, L, x + (int64_t)r0 * h->pN, nr, xt, tt, ex, s) + 1;
        MmOutArgs a{L.d_mm_runit, L.d_mm_ca, L.d_mm_eout, L.d_mm_os, xt, tt, (int)L.mm_n_xch,
                    tiles, nr, L.mm_n_tch, ex, ex + L.mm_n_xch * 16 * tiles, L.d_mm_orow, 16 * tiles, tiles};
        mm_attr((const void *)k_mm_resid, MM_SMEM);
        k_mm_resid<<<(unsigned)(tiles * L.mm_n_runit), MMW * 32, MM_SMEM, s>>>(a, own + (int64_t)r0 * h->pN,
                                                                                           pstride, h->pN);
    }
    return n;
}

} // namespace hm
