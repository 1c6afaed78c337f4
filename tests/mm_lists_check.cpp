// Host-side check of the matrix-instruction products' lists (csrc/hm_lists.h,
// build_mm_lists): on random small blocks with integer values, the two stages are
// walked as the kernels walk them (every pool offset, operand tile and store index in
// bounds, paired loads on even offsets, every T pair written exactly once) and must give
// exactly the directed products' sums.  Prints "ok ..." and exits 0, or the first
// violation and exits 1.
//
// usage: mm_lists_check <seed> <mode> <target>
//   mode 0: random cluster lengths 1..64, dense and low-rank blocks, ranks 1..32
//   mode 1: low-rank only, rank 1;  2: low-rank only, rank 32;  3: no blocks;  4: one dense block
//   mode 5: mode 0 with two T pairs swapped (must FAIL)
#include "hm_lists.h"

#include <cstdio>
#include <cstdlib>
#include <random>

using namespace hm;

static int fail(const char *what)
{
    std::printf("FAIL %s\n", what);
    return 1;
}

int main(int argc, char **argv)
{
    if (argc < 4) return fail("usage");
    const int seed = std::atoi(argv[1]), mode = std::atoi(argv[2]), target = std::atoi(argv[3]);
    std::mt19937 rng(seed);
    auto uni = [&](int lo, int hi) { return std::uniform_int_distribution<int>(lo, hi)(rng); };
    const int ncl = 20;
    std::vector<int> len(ncl), off(ncl);
    for (int i = 0; i < ncl; ++i) { len[i] = uni(1, 64); off[i] = 64 * i; }
    std::vector<Item> items;
    int64_t pool_n = 0;
    auto add = [&](int i, int j, int k) {   // low-rank items have padded (even) lengths, dense ones true lengths
        Item it{pool_n, off[i], off[j], k ? (int)even(len[i]) : len[i], k ? (int)even(len[j]) : len[j], k, 0};
        pool_n += item_elems(it) + (item_elems(it) & 1);
        items.push_back(it);
    };
    if (mode == 4) add(3, 5, 0);
    else if (mode != 3)
        for (int i = 0; i < ncl; ++i)
            for (int j = i + 1; j < ncl; ++j)
                if (uni(0, 3)) add(i, j, mode == 1 ? 1 : mode == 2 ? 32 : uni(0, 2) ? uni(1, 32) : 0);
    const auto by_out = directed_products(items);
    MmLists L;
    if (!build_mm_lists(by_out, target, L)) return fail("build");
    if (mode == 5) std::swap(L.pairs[1].dst, L.pairs[2].dst);
    std::vector<int> pool(pool_n + 2), x(64 * ncl + 2);
    for (int &v : pool) v = uni(-3, 3);
    for (int &v : x) v = uni(-3, 3);
    auto at = [&](int64_t o) -> int {
        if (o < 0 || o >= pool_n) { std::printf("FAIL pool offset %lld\n", (long long)o); std::exit(1); }
        return pool[o];
    };
    // x tiles: zero past the chunk's length
    std::vector<long> xt(L.xch.size() * MM_K, 0), tt(L.n_tch * MM_K, 0);
    for (size_t c = 0; c < L.xch.size(); ++c) {
        if (L.xch[c].off & 1 || L.xch[c].len < 1 || L.xch[c].len > MM_K) return fail("x chunk");
        for (int k = 0; k < L.xch[c].len; ++k) xt[c * MM_K + k] = x[L.xch[c].off + k];
    }
    std::vector<int> written(L.n_tch * (MM_K / 2), 0);
    for (const MmBatch &b : L.batches)
        for (int tile = b.tile0; tile < b.tile0 + b.ntiles; ++tile)
            for (int g = 0; g < 8; ++g) {
                const MmPair &P = L.pairs[4 * (size_t)tile + (g >> 1)];
                const int64_t o = P.w < 0 || ((g & 1) && P.ld == 0) ? -1 : P.w + (g & 1) * (int64_t)P.ld;
                if (o >= 0 && (o & 1)) return fail("odd W row");
                long s = 0;
                for (int k = 0; k < b.klen; ++k)
                    if (o >= 0) s += (long)at(o + k) * xt[((size_t)b.xg0 + k / MM_K) * MM_K + k % MM_K];
                if (P.dst < 0) continue;
                tt[2 * (size_t)P.dst + (g & 1)] = s;
                written[P.dst] += g & 1;
            }
    for (int w : written)
        if (w != 1) return fail("a T pair not written once");
    auto output = [&](const std::vector<MmUnit> &units) {
        std::vector<long> z(64 * ncl, 0);
        for (const MmUnit &u : units)
            for (int c = u.c0; c < u.c1; ++c) {
                const MmChunk &C = L.chunks[c];
                for (int i = 0; i < C.olen; ++i)
                    for (int k = 0; k < MM_K; ++k) {
                        long v = 0;
                        if (C.kind == 2) {
                            const int64_t row = L.rows[C.src + k];
                            if (row >= 0) v = at(row + i) * tt[(size_t)C.a * MM_K + k];
                        } else if (k < C.klen) {
                            if (C.kind == 0 && ((C.src | C.ld) & 1)) { std::printf("FAIL odd natural row\n"); std::exit(1); }
                            v = (long)at(C.kind == 0 ? C.src + (int64_t)i * C.ld + k : C.src + (int64_t)k * C.ld + i) *
                                xt[(size_t)C.a * MM_K + k];
                        }
                        if (i >= u.mlen && v) { std::printf("FAIL output past the unit\n"); std::exit(1); }
                        z[u.out0 + i] += v;
                    }
            }
        return z;
    };
    // the operand streams: every chunk's and batch's tiles one after another, units start at their first chunk
    int64_t pos = 0;
    for (const MmChunk &c : L.chunks) {
        if (c.pos != pos || c.tiles < 1 || c.olen > 8 * c.tiles || c.cl < 0 || c.cl >= L.n_cl) return fail("chunk stream");
        pos += c.tiles;
    }
    if (pos != L.n_out) return fail("output stream length");
    pos = 0;
    for (const MmBatch &b : L.batches) {
        if (b.pos != pos) return fail("batch stream");
        pos += (int64_t)b.ntiles * ((b.klen + MM_K - 1) / MM_K);
    }
    if (pos != L.n_w) return fail("stage-1 stream length");
    for (const auto *us : {&L.units, &L.units2, &L.runits})
        for (const MmUnit &u : *us)
            if (u.c0 >= u.c1 || u.pos != L.chunks[u.c0].pos || L.chunks[u.c0].cl != u.cl || L.chunks[u.c1 - 1].cl != u.cl ||
                (u.mlen + 7) / 8 != L.chunks[u.c0].tiles)
                return fail("unit stream");
    // every chunk of a cluster in exactly one unit, parts numbered within the cluster
    for (const auto *us : {&L.units, &L.units2, &L.runits}) {
        std::vector<int> seen(L.chunks.size(), 0);
        for (const MmUnit &u : *us) {
            for (int c = u.c0; c < u.c1; ++c) seen[c]++;
            if (u.cl < 0 || u.cl >= L.n_cl || u.part < 0 || (us == &L.runits && u.part >= L.parts)) return fail("unit");
        }
        for (int n : seen)
            if (n != 1) return fail("a chunk not in exactly one unit");
    }
    std::vector<long> want(64 * ncl, 0);
    for (const Item &it : items)
        for (int i = 0; i < it.m; ++i)
            for (int j = 0; j < it.n; ++j) {
                long v = 0;
                const int64_t lm = even(it.m), ln = even(it.n);
                if (it.k == 0) v = pool[it.off + i * ln + j];
                for (int l = 0; l < it.k; ++l) v += (long)pool[it.off + l * lm + i] * pool[it.off + it.k * lm + l * ln + j];
                want[it.row0 + i] += v * x[it.col0 + j];
                want[it.col0 + j] += v * x[it.row0 + i];
            }
    if (output(L.units) != want) return fail("product units' sums");
    if (output(L.units2) != want) return fail("coarse product units' sums");
    if (output(L.runits) != want) return fail("residual units' sums");
    // the scale sets: every directed product once, its pairs and T rows where the stages use them
    size_t np = 0;
    for (auto &kv : by_out) np += kv.second.size();
    if (L.sets.size() != np) return fail("number of scale sets");
    for (const MmSet &s : L.sets)
        for (int l = 0; l < s.rank; ++l) {
            const MmPair &P = L.pairs[s.p0 + l / 2];
            if (P.w + (l & 1) * (int64_t)P.ld != s.w + (int64_t)l * s.w_ld) return fail("scale set W row");
            if (mode != 5 && P.dst != s.t0 + l / 2) return fail("scale set T pair");
            if (L.rows[2 * (size_t)(s.t0 + l / 2) + (l & 1)] != s.y + (int64_t)l * s.y_ld) return fail("scale set Y row");
        }
    std::printf("ok %zu chunks %zu units %zu runits %lld T chunks\n", L.chunks.size(), L.units.size(), L.runits.size(),
                (long long)L.n_tch);
    return 0;
}
