// Work lists of the block products: the host logic that orders the stored blocks
// for the kernels (plain C++, no CUDA types, so that the CPU tests compile it with
// the host compiler; hm_internal.h includes it).
//  - Item: one stored block, the work item of the product and residual kernels.
//  - TcProd / TcUnit: the directed products of the small blocks (each block gives two,
//    eq. 6 and eq. 8 with the half storage of §III of arxiv 2307.03968), grouped by
//    output cluster.
//  - TcOp / TcBatch / XChunk: the tensor-core product's two launches (k_mrhs_tc.cu).
#pragma once

#include <algorithm>
#include <climits>
#include <cstdint>
#include <map>
#include <utility>
#include <vector>

#ifdef __CUDACC__
#define HM_HD __host__ __device__
#else
#define HM_HD
#endif

namespace hm {

constexpr int MRHS_MAX_DIM = 64;    // largest block side of the multi-RHS product kernel
constexpr int MRHS_MAX_RANK = 32;   // largest rank of a low-rank block it takes
constexpr int TC_MAX_DIM = MRHS_MAX_DIM;    // the tensor-core product takes the same small items
constexpr int TC_MAX_RANK = MRHS_MAX_RANK;
constexpr int TC_UNIT_CHUNKS = 64;  // K chunks (of 8) a tensor-core work unit sums in tensor memory

// One stored block = one work item of the product kernels (32 bytes).
struct Item {
    int64_t off;    // complex-element offset into the pool
    int32_t row0;   // padded-tree offset of the row cluster
    int32_t col0;   // padded-tree offset of the column cluster
    int32_t m, n;   // padded cluster lengths (dense: m = true rows, n = true cols)
    int32_t k;      // rank; 0 = dense block
    int32_t pad;    // offset of the block's partial slots (row side, then column side)
};
static_assert(sizeof(Item) == 32, "Item layout");

// One directed product of a small stored block into an output cluster (the
// owner-computes residual, k_resid_own.cu): Z_out += B X_in with B the block (dense,
// read row-major or transposed) or, for a low-rank block, Y (W X_in) with the
// input-side factor W read row-major (rank rows) and the output-side factor Y
// read transposed.
struct TcProd {
    int64_t b_off;   // complex offset of the block (dense) or of W (low-rank)
    int64_t y_off;   // complex offset of Y (low-rank)
    int32_t in0;     // padded-tree offset of the input cluster
    int32_t klen;    // input length (K of the dense product and of stage 1)
    int32_t rank;    // 0 = dense
    int32_t b_ld;    // row stride of the block / of W
    int32_t y_ld;    // row stride of Y as stored (rank rows)
    int32_t trans;   // dense: 1 = element (out i, in j) is block[j][i] (the mirror product)
    int32_t olen;    // output length of this product
    int32_t xg0;     // first K chunk of the input cluster in the level's split-x chunk list
};
static_assert(sizeof(TcProd) == 48, "TcProd layout");
// a work unit: products [p0, p1) into the output cluster at out0 (mlen = largest olen)
struct TcUnit { int32_t out0, mlen, p0, p1; };

// The tensor-core product (k_mrhs_tc.cu) in two launches.  The first runs stage 1 of
// every low-rank directed product, T = W X_in, batched over the products that share
// an input cluster (their W rows stacked along N); it stores T in chunks of 8 rank
// rows (TC_T_CHUNK floats per chunk and RHS tile).  The second runs, per output
// cluster, the dense products and the second stages Y T, which read T back.
constexpr int TC_T_CHUNK = 2 * 128 * 8;   // floats of one T chunk: Re and Im planes of 128 RHS x 8 rank rows
// one operation of the second launch
struct TcOp {
    int64_t src;     // complex offset of the dense block, or of Y (low-rank second stage)
    int64_t t0;      // low-rank: first T chunk of the product (per RHS tile)
    int32_t kind;    // 0 dense (element (out i, in j) = block[i][j]), 1 dense mirror (= block[j][i]), 2 Y T
    int32_t klen;    // K length: the input length (dense) or the rank
    int32_t ld;      // row stride of the block or of Y as stored (rank rows)
    int32_t olen;    // output length
    int32_t xg0;     // dense: first split-x chunk of the input cluster
    int32_t pad;
};
static_assert(sizeof(TcOp) == 40, "TcOp layout");
// a batch of the first launch: stacked rows [row0, row0 + nrows) (nrows a multiple of
// 8, at most 64) of the row table, all over one input cluster (split-x chunks from xg0,
// K length klen); each row's W offset (-1: a zero row) is in the row table, each group
// of 8 rows' T chunk in the chunk table (index row / 8)
struct TcBatch { int32_t xg0, klen, row0, nrows; };
// a K chunk of an input cluster for the split x: padded-tree offset and valid length (<= 8)
struct XChunk { int32_t off, len; };

HM_HD inline int64_t even(int64_t v) { return (v + 1) & ~int64_t(1); }

HM_HD inline int64_t item_elems(const Item &it)
{
    if (it.k == 0) return int64_t(it.m) * even(it.n);
    return int64_t(it.k) * (even(it.m) + even(it.n));
}

// The directed products of the small items: every item gives two (into its row
// cluster and, mirrored, into its column cluster), grouped by output cluster.
inline std::map<int32_t, std::vector<TcProd>> directed_products(const std::vector<Item> &small)
{
    std::map<int32_t, std::vector<TcProd>> by_out;
    auto add = [&](int32_t out0, const TcProd &p) {
        if (p.klen > 0 && p.olen > 0) by_out[out0].push_back(p);
    };
    for (const Item &it : small) {
        if (it.k == 0) {
            const int32_t ld = (int32_t)even(it.n);
            add(it.row0, TcProd{it.off, 0, it.col0, it.n, 0, ld, 0, 0, it.m, 0});
            add(it.col0, TcProd{it.off, 0, it.row0, it.m, 0, ld, 0, 1, it.n, 0});
        } else {
            const int32_t lm = (int32_t)even(it.m), ln = (int32_t)even(it.n);
            const int64_t uoff = it.off, voff = it.off + (int64_t)it.k * lm;
            add(it.row0, TcProd{voff, uoff, it.col0, it.n, it.k, ln, lm, 0, it.m, 0});   // U (V x_J)
            add(it.col0, TcProd{uoff, voff, it.row0, it.m, it.k, lm, ln, 0, it.n, 0});   // V^T (U^T x_I)
        }
    }
    return by_out;
}

// The owner-computes residual's list: one unit per output cluster (every output row
// summed by one CTA in a fixed order), largest first.
inline void build_owner_lists(const std::map<int32_t, std::vector<TcProd>> &by_out, std::vector<TcUnit> &runits,
                              std::vector<TcProd> &rprods)
{
    auto cost = [](const TcProd &p) {
        return (int64_t)((p.klen + 7) / 8) + (p.rank > 0 ? (int64_t)((p.rank + 7) / 8) : 0);
    };
    struct R { TcUnit u; int64_t c; const std::vector<TcProd> *p; };
    std::vector<R> rs;
    for (auto &kv : by_out) {
        R r{TcUnit{kv.first, 0, 0, 0}, 0, &kv.second};
        for (const TcProd &p : kv.second) { r.u.mlen = std::max(r.u.mlen, p.olen); r.c += cost(p); }
        rs.push_back(r);
    }
    std::stable_sort(rs.begin(), rs.end(), [](const R &a, const R &b) { return a.c > b.c; });
    runits.clear();
    rprods.clear();
    for (R &r : rs) {
        r.u.p0 = (int32_t)rprods.size();
        rprods.insert(rprods.end(), r.p->begin(), r.p->end());
        r.u.p1 = (int32_t)rprods.size();
        runits.push_back(r.u);
    }
}

// Whether the clusters of a level's small items (sides of at most MRHS_MAX_DIM, padded positions below
// pN) are disjoint or the same; at one start the longest counts.  The clusters of one tree level are;
// a user's own blocks may couple, on the same level, a leaf and a union that holds it.  The
// owner-computes residuals store each cluster's sums, so two clusters that share rows would
// overwrite each other's.
inline bool disjoint_clusters(const std::vector<Item> &items, int64_t pN)
{
    std::vector<int32_t> len((size_t)pN, 0);
    for (const Item &it : items)
        if (it.m <= MRHS_MAX_DIM && it.n <= MRHS_MAX_DIM && it.k <= MRHS_MAX_RANK) {
            len[it.row0] = std::max(len[it.row0], it.m);
            len[it.col0] = std::max(len[it.col0], it.n);
        }
    int64_t end = 0;
    for (int64_t p = 0; p < pN; ++p)
        if (len[p] > 0) {
            if (p < end) return false;
            end = p + len[p];
        }
    return true;
}

// The owner units cut into parts of about equal cost, so that a call has `target` units a
// right-hand-side group where there are fewer clusters than that (each part sums into an array of
// its own, which the gather adds in order), parts of at least 8 products; returns the parts.
struct RcUnit { int32_t out0, mlen, p0, p1, part; };
inline int split_owner_units(const std::vector<TcUnit> &units, const std::vector<TcProd> &prods, int64_t target,
                             std::vector<RcUnit> &out)
{
    auto cost = [](const TcProd &p) { return (int64_t)(p.rank > 0 ? 2 * p.rank + 24 : p.klen + 16); };
    const int64_t want = units.empty() ? 1 : (target + (int64_t)units.size() - 1) / (int64_t)units.size();
    int parts = 1;
    std::vector<std::pair<int64_t, RcUnit>> rs;
    for (const TcUnit &u : units) {
        const int n = (int)std::max<int64_t>(1, std::min<int64_t>(want, (u.p1 - u.p0) / 8));
        int64_t total = 0, run = 0, from = 0;
        for (int32_t p = u.p0; p < u.p1; ++p) total += cost(prods[p]);
        RcUnit r{u.out0, u.mlen, u.p0, u.p0, 0};
        for (int32_t p = u.p0; p < u.p1; ++p) {
            run += cost(prods[p]);
            r.p1 = p + 1;
            if (p + 1 == u.p1 || (r.part + 1 < n && run * n >= total * (r.part + 1))) {
                rs.push_back({run - from, r});
                parts = std::max(parts, r.part + 1);
                r.p0 = p + 1;
                ++r.part;
                from = run;
            }
        }
    }
    std::stable_sort(rs.begin(), rs.end(), [](const auto &a, const auto &b) { return a.first > b.first; });
    out.clear();
    for (const auto &r : rs) out.push_back(r.second);
    return parts;
}

// The tensor-core product's lists (k_mrhs_tc.cu), two launches.
//  - Stage 1 of every low-rank directed product, T = W X_in (W = V forward, U^T mirrored),
//    is batched over the products that share an input cluster: each product takes
//    roundup8(rank) stacked rows (rows past its rank are zero) and as many T chunks, and a
//    batch stacks up to 64 rows, so one K chunk of split x feeds MMAs of N up to 128.
//  - The second launch takes, per output cluster, the dense products and the second
//    stages Y T (Y = U forward, V^T mirrored; T read back by chunk), cut into units of at
//    most TC_UNIT_CHUNKS K chunks (units of one cluster add into z with atomics) and sorted
//    by cost, largest first, so that the persistent CTAs taking units in turn stay balanced.
// Returns false when a list would break an index bound the kernels rely on.
struct TcLists {
    std::vector<TcUnit> units;
    std::vector<TcOp> ops;
    std::vector<XChunk> xch;
    std::vector<TcBatch> batches;
    std::vector<int64_t> rows;
    std::vector<int32_t> tchunks;
    int64_t n_tchunk = 0;
};
inline bool build_tc_lists(const std::map<int32_t, std::vector<TcProd>> &by_out, TcLists &T)
{
    // K chunks of the input clusters (each cluster's longest input length)
    std::map<int32_t, int32_t> in_len;
    for (auto &kv : by_out)
        for (const TcProd &p : kv.second) in_len[p.in0] = std::max(in_len[p.in0], p.klen);
    std::map<int32_t, int32_t> in_g0;
    T.xch.clear();
    for (auto &kv : in_len) {
        in_g0[kv.first] = (int32_t)T.xch.size();
        for (int32_t c = 0; c < kv.second; c += 8) T.xch.push_back(XChunk{kv.first + c, std::min(8, kv.second - c)});
    }
    // stage-1 jobs by (input cluster, K length), each with its first T chunk
    struct Job { int64_t w_off; int32_t w_ld, rank; int64_t t0; };
    std::map<std::pair<int32_t, int32_t>, std::vector<Job>> by_in;
    T.n_tchunk = 0;
    // second-launch operations per output cluster
    auto chunks = [](int32_t klen) { return (int64_t)((klen + 7) / 8); };
    const int64_t cap = TC_UNIT_CHUNKS;
    struct U { TcUnit u; int64_t c; std::vector<TcOp> p; };
    std::vector<U> us;
    for (auto &kv : by_out) {
        int32_t mlen = 0;
        for (const TcProd &p : kv.second) mlen = std::max(mlen, p.olen);
        U cur{TcUnit{kv.first, mlen, 0, 0}, 0, {}};
        for (const TcProd &p : kv.second) {
            TcOp op{};
            op.olen = p.olen;
            if (p.rank == 0) {
                op.src = p.b_off;
                op.kind = p.trans ? 1 : 0;
                op.klen = p.klen;
                op.ld = p.b_ld;
                op.xg0 = in_g0[p.in0];
            } else {
                op.src = p.y_off;
                op.t0 = T.n_tchunk;
                op.kind = 2;
                op.klen = p.rank;
                op.ld = p.y_ld;
                by_in[{p.in0, p.klen}].push_back(Job{p.b_off, p.b_ld, p.rank, T.n_tchunk});
                T.n_tchunk += chunks(p.rank);
            }
            // Units of at most TC_UNIT_CHUNKS K chunks: the tensor cores' FP32 accumulator loses
            // a little on every MMA it adds into a large running sum (measured: the product's
            // error grows in proportion to the chunks summed in tensor memory, 7.4e-6 relative
            // at 256 chunks, 1.9e-6 at 64, 5.4e-7 at 16 on 60-unknown leaves), so a unit's sum
            // leaves tensor memory (added into z in FP32) every TC_UNIT_CHUNKS chunks.
            if (cur.c > 0 && cur.c + chunks(op.klen) > cap) {
                us.push_back(cur);
                cur.c = 0;
                cur.p.clear();
            }
            cur.p.push_back(op);
            cur.c += chunks(op.klen);
        }
        if (!cur.p.empty()) us.push_back(cur);
    }
    std::stable_sort(us.begin(), us.end(), [](const U &a, const U &b) { return a.c > b.c; });
    T.units.clear();
    T.ops.clear();
    for (U &x : us) {
        x.u.p0 = (int32_t)T.ops.size();
        T.ops.insert(T.ops.end(), x.p.begin(), x.p.end());
        x.u.p1 = (int32_t)T.ops.size();
        T.units.push_back(x.u);
    }
    // stage-1 batches of at most 64 stacked rows
    T.batches.clear();
    T.rows.clear();
    T.tchunks.clear();
    for (auto &kv : by_in) {
        const int32_t xg0 = in_g0[kv.first.first], klen = kv.first.second;
        TcBatch b{xg0, klen, (int32_t)T.rows.size(), 0};
        for (const Job &j : kv.second) {
            const int32_t k8 = (j.rank + 7) & ~7;
            if (b.nrows + k8 > 64) {
                T.batches.push_back(b);
                b = TcBatch{xg0, klen, (int32_t)T.rows.size(), 0};
            }
            for (int32_t l = 0; l < k8; ++l) T.rows.push_back(l < j.rank ? j.w_off + (int64_t)l * j.w_ld : -1);
            for (int32_t g = 0; g < k8 / 8; ++g) T.tchunks.push_back((int32_t)(j.t0 + g));
            b.nrows += k8;
        }
        if (b.nrows > 0) T.batches.push_back(b);
    }
    // the bounds the kernels index by
    if (T.n_tchunk > INT32_MAX || (int64_t)T.rows.size() > INT32_MAX || T.ops.size() > (size_t)INT32_MAX) return false;
    if ((int64_t)T.tchunks.size() * 8 != (int64_t)T.rows.size()) return false;
    for (const TcBatch &b : T.batches)
        if (b.nrows <= 0 || b.nrows > 64 || (b.nrows & 7) || b.row0 < 0 || (b.row0 & 7) ||
            b.row0 + (int64_t)b.nrows > (int64_t)T.rows.size() ||
            b.xg0 + chunks(b.klen) > (int64_t)T.xch.size())
            return false;
    for (int32_t t : T.tchunks)
        if (t < 0 || t >= T.n_tchunk) return false;
    for (const TcOp &o : T.ops) {
        if (o.olen <= 0 || o.olen > TC_MAX_DIM || o.klen <= 0) return false;
        if (o.kind == 2 ? (o.klen > TC_MAX_RANK || o.t0 + chunks(o.klen) > T.n_tchunk)
                        : (o.klen > TC_MAX_DIM || o.xg0 + chunks(o.klen) > (int64_t)T.xch.size()))
            return false;
    }
    for (const TcUnit &u : T.units)
        if (u.mlen > TC_MAX_DIM || u.p0 < 0 || u.p1 <= u.p0 || u.p1 > (int32_t)T.ops.size()) return false;
    return true;
}

// The matrix-instruction products' lists (k_mm.cu): the small items of a level as two
// dense matrix products.
//  - Stage 1, per input cluster J: T = W X_J with the W rows (rank rows) of every low-rank
//    directed product from J stacked, two at a time (MmPair), eight to a tile; MmBatch is
//    a run of tiles over one input cluster.
//  - Output, per output cluster: Z = [B_1 B_2 ... Y_1 Y_2 ...] [X; X; ... T_1; T_2; ...], K in
//    chunks of 16 (MmChunk): chunks of the dense products over split-x chunks, then the rank
//    rows of all low-rank products one after another (pairs, T in that order, so that no
//    rank is padded beyond an even number of rows), MmUnit a run of chunks.
constexpr int MM_K = 16;            // K per chunk (one matrix instruction)
struct MmChunk {
    int64_t src;     // kind 0: element (out 0, k 0); 1: the same (rows are K); 2: first of the chunk's 16 row offsets
    int32_t a;       // split-x chunk (kinds 0, 1) or T chunk (2)
    int32_t ld;      // row stride (kinds 0, 1)
    int16_t kind;    // 0 dense, element (i, k) = src[i ld + k]; 1 dense mirrored, src[k ld + i]; 2 rank rows, pool[row[k] + i]
    int16_t klen;    // valid K of the chunk
    int16_t olen;    // valid outputs
    int16_t tiles;   // tiles of 8 outputs of its cluster
    int32_t cl;      // its output cluster
    int32_t pos;     // its first tile in the operand stream
};
static_assert(sizeof(MmChunk) == 32, "MmChunk layout");
// chunks [c0, c1) of output cluster cl, the first at tile pos of the stream; part: the unit's
// index among the cluster's units
struct MmUnit { int32_t out0, mlen, c0, c1, cl, part, pos; };
struct MmPair { int64_t w; int32_t ld, dst; };   // W rows at w and w + ld (ld 0: one row; w -1: none) -> T pair dst (-1: no store)
struct MmBatch { int32_t xg0, klen, tile0, ntiles, pos; };   // pos: first 8 x 16 tile in the stream (chunk fastest)
struct MmSet {       // one directed product, for the scales: rank > 0: W (rank x klen) and Y (rank x olen); 0: the block at w
    int64_t w, y;
    int32_t w_ld, y_ld, rank, wlen, ylen;   // rank 0: y_ld = rows
    int32_t t0, p0, cl;  // first T pair, first stage-1 pair, output cluster
};
struct MmLists {
    std::vector<MmChunk> chunks;
    std::vector<int64_t> rows;       // 16 per T chunk: pool offsets of the Y rows (-1: none)
    std::vector<MmUnit> units, units2, runits;
    std::vector<MmPair> pairs;       // four to a tile
    std::vector<MmBatch> batches;
    std::vector<XChunk> xch;
    std::vector<MmSet> sets;
    int64_t n_tch = 0;               // T chunks
    int64_t n_out = 0, n_w = 0;      // 8 x 16 tiles of the output and of the stage-1 stream
    int32_t n_cl = 0, parts = 1;     // output clusters; residual units of a cluster, at most
};

// target: work units wanted for one tile of right-hand sides (a few CTAs per SM)
inline bool build_mm_lists(const std::map<int32_t, std::vector<TcProd>> &by_out, int64_t target, MmLists &L)
{
    std::map<int32_t, int32_t> in_len, in_g0;
    for (auto &kv : by_out)
        for (const TcProd &p : kv.second) {
            int32_t &v = in_len[p.in0];
            v = std::max(v, p.klen);
        }
    for (auto &kv : in_len) {
        in_g0[kv.first] = (int32_t)L.xch.size();
        for (int32_t c = 0; c < kv.second; c += MM_K) L.xch.push_back(XChunk{kv.first + c, std::min(MM_K, kv.second - c)});
    }
    std::map<std::pair<int32_t, int32_t>, std::vector<MmPair>> by_in;
    std::map<std::pair<int32_t, int32_t>, std::vector<size_t>> sets_in;    // sets in the order of their pairs
    struct C { int32_t out0, mlen, c0, c1; };
    std::vector<C> cls;
    for (auto &kv : by_out) {
        C c{kv.first, 0, (int32_t)L.chunks.size(), 0};
        const int32_t cl = (int32_t)cls.size();
        for (const TcProd &p : kv.second) {
            c.mlen = std::max(c.mlen, p.olen);
            if (p.rank > 0) continue;
            for (int32_t k = 0; k < p.klen; k += MM_K)
                L.chunks.push_back(MmChunk{p.b_off + (p.trans ? (int64_t)k * p.b_ld : k), in_g0[p.in0] + k / MM_K, p.b_ld,
                                           (int16_t)(p.trans ? 1 : 0), (int16_t)std::min(MM_K, p.klen - k), (int16_t)p.olen, 0, cl, 0});
            L.sets.push_back(MmSet{p.b_off, 0, p.b_ld, p.trans ? p.klen : p.olen, 0, p.trans ? p.olen : p.klen, 0, 0, 0, cl});
        }
        // rank rows: pairs in product order; a chunk holds rows of one output length
        int fill = MM_K, olen = -1;
        std::pair<int32_t, int32_t> last{0, 0};
        auto pad = [&] {
            for (; fill < MM_K; fill += 2)
                by_in[last].push_back(MmPair{-1, 0, (int32_t)((L.n_tch - 1) * (MM_K / 2) + fill / 2)});
        };
        for (const TcProd &p : kv.second) {
            if (p.rank == 0) continue;
            if (p.olen != olen) pad();
            olen = p.olen;
            MmSet st{p.b_off, p.y_off, p.b_ld, p.y_ld, p.rank, p.klen, p.olen, 0, 0, cl};
            last = {p.in0, p.klen};
            std::vector<MmPair> &in = by_in[last];
            st.p0 = (int32_t)in.size();
            for (int32_t l = 0; l < p.rank; l += 2) {
                if (fill == MM_K) {
                    L.chunks.push_back(MmChunk{(int64_t)L.rows.size(), (int32_t)L.n_tch, 0, 2, MM_K, (int16_t)p.olen, 0, cl, 0});
                    L.rows.insert(L.rows.end(), MM_K, -1);
                    ++L.n_tch;
                    fill = 0;
                }
                const int32_t dst = (int32_t)((L.n_tch - 1) * (MM_K / 2) + fill / 2);
                if (l == 0) st.t0 = dst;
                in.push_back(MmPair{p.b_off + (int64_t)l * p.b_ld, l + 1 < p.rank ? p.b_ld : 0, dst});
                int64_t *row = &L.rows[(size_t)dst * 2];
                row[0] = p.y_off + (int64_t)l * p.y_ld;
                if (l + 1 < p.rank) row[1] = row[0] + p.y_ld;
                fill += 2;
            }
            sets_in[last].push_back(L.sets.size());
            L.sets.push_back(st);
        }
        pad();
        c.c1 = (int32_t)L.chunks.size();
        for (int32_t q = c.c0; q < c.c1; ++q) {
            L.chunks[q].tiles = (int16_t)((c.mlen + 7) / 8);
            L.chunks[q].pos = (int32_t)L.n_out;
            L.n_out += L.chunks[q].tiles;
        }
        if (L.n_out > INT32_MAX) return false;
        cls.push_back(c);
    }
    if (L.n_tch > INT32_MAX / MM_K || L.chunks.size() > (size_t)INT32_MAX) return false;
    L.n_cl = (int32_t)cls.size();
    // units: enough for the SMs; the residual keeps its sums per unit ([part][RHS][pN]), so few a cluster
    const int64_t n_ch = (int64_t)L.chunks.size();
    // product units of at most cap chunks: fine ones, enough for the SMs with one tile of right-hand
    // sides; coarse ones where more tiles give the CTAs, 32 chunks for each of the K groups that share
    // a unit there (k_mm_out: 8 warps, 16 outputs a warp, two groups of right-hand sides)
    const int64_t cap = std::min<int64_t>(256, std::max<int64_t>(8, (n_ch + target - 1) / target));
    L.parts = (int32_t)std::min<int64_t>(8, std::max<int64_t>(1, (target + L.n_cl - 1) / std::max<int32_t>(L.n_cl, 1)));
    for (int32_t i = 0; i < L.n_cl; ++i) {
        const C &c = cls[i];
        const int64_t n = c.c1 - c.c0;
        auto cut = [&](std::vector<MmUnit> &us, int64_t np) {
            for (int64_t q = 0; q < np; ++q)
                us.push_back(MmUnit{c.out0, c.mlen, (int32_t)(c.c0 + n * q / np), (int32_t)(c.c0 + n * (q + 1) / np), i, (int32_t)q, 0});
        };
        cut(L.units, (n + cap - 1) / cap);
        const int64_t cap2 = std::max<int64_t>(cap, 32 * (8 / (2 * ((c.mlen + 15) / 16))));
        cut(L.units2, (n + cap2 - 1) / cap2);
        cut(L.runits, std::max<int64_t>(1, std::min<int64_t>(L.parts, (n + 7) / 8)));
    }
    for (auto *us : {&L.units, &L.units2, &L.runits})
        for (MmUnit &u : *us) u.pos = u.c0 < u.c1 ? L.chunks[u.c0].pos : 0;
    auto longest = [](const MmUnit &a, const MmUnit &b) { return a.c1 - a.c0 > b.c1 - b.c0; };
    std::stable_sort(L.units.begin(), L.units.end(), longest);
    std::stable_sort(L.units2.begin(), L.units2.end(), longest);
    std::stable_sort(L.runits.begin(), L.runits.end(), longest);
    // stage 1: whole tiles of four pairs per input cluster, batches of at most 32 tiles
    for (auto &kv : by_in) {
        std::vector<MmPair> &v = kv.second;
        const int32_t base = (int32_t)L.pairs.size();
        for (size_t q : sets_in[kv.first]) L.sets[q].p0 += base;
        while (v.size() & 3) v.push_back(MmPair{-1, 0, -1});
        const int32_t t0 = base / 4, nt = (int32_t)(v.size() / 4);
        const int32_t nch = (kv.first.second + MM_K - 1) / MM_K;
        for (int32_t t = 0; t < nt; t += 32) {
            L.batches.push_back(MmBatch{in_g0[kv.first.first], kv.first.second, t0 + t, std::min(32, nt - t), (int32_t)L.n_w});
            L.n_w += (int64_t)nch * std::min(32, nt - t);
        }
        if (L.n_w > INT32_MAX) return false;
        L.pairs.insert(L.pairs.end(), v.begin(), v.end());
    }
    // the bounds the kernels index by
    const int64_t n_x = (int64_t)L.xch.size();
    for (const MmChunk &c : L.chunks)
        if (c.klen < 1 || c.klen > MM_K || c.olen < 1 || c.olen > MRHS_MAX_DIM || c.a < 0 ||
            c.a >= (c.kind == 2 ? L.n_tch : n_x) || (c.kind == 2 && c.src + MM_K > (int64_t)L.rows.size()))
            return false;
    for (const MmPair &p : L.pairs)
        if (p.dst >= L.n_tch * (MM_K / 2)) return false;
    for (const MmBatch &b : L.batches)
        if (b.klen < 1 || b.klen > MRHS_MAX_DIM || b.xg0 + (b.klen + MM_K - 1) / MM_K > n_x ||
            4 * ((int64_t)b.tile0 + b.ntiles) > (int64_t)L.pairs.size())
            return false;
    for (const MmUnit &u : L.units)
        if (u.mlen > MRHS_MAX_DIM || u.c0 > u.c1) return false;
    return true;
}

// The FP32 product gives each item of its list to one warp, so long blocks are cut: a dense
// block of more than PROD_PANEL rows into row panels (rows [r, r + mr) of a row-major block are
// themselves a dense item of the same row stride), a low-rank block longer than 64 into panels of
// PROD_RANK rank rows (their sum is the block's product; the kernel works in steps of that many
// rank rows anyway, so the panels add no memory traffic).  A low-rank item's pad is half the
// distance (m and n are even) from its U^T panel to its V panel (panel_voff).
// (30,720-unknown sphere, level 2: 80 blocks of 480 x 480 and more took 152 us on 80 warps.)
constexpr int PROD_PANEL = 64;
constexpr int PROD_RANK = 8;
// low-rank blocks longer than 64 x 64
inline bool wide_item(const Item &it) { return it.k > 0 && (it.m > 64 || it.n > 64); }
// of those, the ones whose panels fill a CTA in the product (its 8 warps take 64 columns each).  The
// panels of shorter ones stay with the warps: 24,120 unknowns in leaves of 95, 125 us a solve (a
// CTA a panel 152, a whole block a warp 145) and 394 us with four right-hand sides (525, 418); 4,720
// in leaves of 74, 47 us (55, 46)
constexpr int PROD_CTA_LEN = 256;
inline bool cta_item(const Item &it) { return it.k > 0 && (it.m > PROD_CTA_LEN || it.n > PROD_CTA_LEN); }
HM_HD inline int64_t panel_voff(const Item &it) { return 2 * (int64_t)(uint32_t)it.pad; }
inline void product_panels(const std::vector<Item> &in, std::vector<Item> &out)
{
    for (const Item &it : in) {
        const int32_t step = it.k == 0 ? PROD_PANEL : wide_item(it) ? PROD_RANK : it.k;
        const int32_t len = it.k == 0 ? it.m : it.k;
        for (int32_t r = 0; r < len; r += step) {
            Item q = it;
            const int32_t c = std::min(step, len - r);
            if (it.k == 0) {
                q.off = it.off + (int64_t)r * even(it.n);
                q.row0 = it.row0 + r;
                q.m = c;
            } else {
                q.off = it.off + (int64_t)r * it.m;
                q.pad = (int32_t)(uint32_t)(((int64_t)(it.k - r) * it.m + (int64_t)r * it.n) / 2);
                q.k = c;
            }
            out.push_back(q);
        }
    }
}

// items reordered for a persistent kernel whose nw warps take items t, t + nw, ...:
// sorted by cost, largest first, and every odd round of nw reversed (a snake), so that
// the warps' sums match.  Cost of the product: stored bytes plus a fixed 2 KB for the
// per-block latencies; of the FP64-class residual (instruction-bound): about 39 lane
// instructions per stored element of a dense block, 52 of a low-rank one, plus 3,000.
inline int64_t product_cost(const Item &it) { return item_elems(it) * 8 + 2048; }
inline int64_t residual_cost(const Item &it) { return item_elems(it) * (it.k == 0 ? 39 : 52) + 3000; }
template <class Cost>
inline std::vector<Item> balanced_order(const std::vector<Item> &in, int64_t nw, Cost cost)
{
    std::vector<Item> v = in;
    std::stable_sort(v.begin(), v.end(), [&](const Item &a, const Item &b) { return cost(a) > cost(b); });
    const int64_t n = (int64_t)v.size();
    nw = std::min<int64_t>(std::max<int64_t>(nw, 1), std::max<int64_t>(n, 1));
    std::vector<Item> out(v.size());
    for (int64_t t = 0; t < n; ++t) {
        const int64_t q = t / nw, p = t % nw, rem = std::min<int64_t>(nw, n - q * nw);
        out[t] = v[q * nw + ((q & 1) ? rem - 1 - p : p)];
    }
    return out;
}

} // namespace hm
