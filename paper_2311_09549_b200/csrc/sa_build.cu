// Host-side construction of the compressed levels (Section 2.1 of the paper: CSR / CSF as a
// tree of levels, arrays named pos / crd / vals as in Fig. 1b) and of the load-balancing work
// lists (nonzero-balanced pieces of slices, fibers and rows) the kernels consume.
#include <algorithm>
#include <atomic>
#include <cstring>
#include <functional>
#include <iterator>
#include <memory>
#include <new>
#include <omp.h>

#include "sa_internal.h"

namespace {

int bits_for(int64_t dim)
{
    int b = 1;
    while ((int64_t(1) << b) < dim) ++b;
    return b;
}

// Stable LSD radix sort of (key, idx) pairs on the low `total_bits` bits, 11 bits per pass.  The second pair of buffers
// is scratch; the sorted pairs end up in keys / idx.  (Buffers that are filled in parallel are allocated without being
// set to zero first: the one thread that would do that takes as long as a pass of the sort.)
void radix_sort(std::unique_ptr<uint64_t[]> &keys, std::unique_ptr<uint32_t[]> &idx, size_t n, int total_bits)
{
    if (n < 2) return;
    constexpr int DB = 11, NB = 1 << DB;
    const int passes = (total_bits + DB - 1) / DB;
    std::unique_ptr<uint64_t[]> k2(new uint64_t[n]);
    std::unique_ptr<uint32_t[]> i2(new uint32_t[n]);
    const int nt = std::max(1, omp_get_max_threads());
    std::vector<size_t> hist(size_t(nt) * NB);
    for (int pass = 0; pass < passes; ++pass) {
        const int shift = pass * DB;
        const uint64_t *ks = keys.get();
        const uint32_t *is = idx.get();
        uint64_t *kd = k2.get();
        uint32_t *id = i2.get();
#pragma omp parallel num_threads(nt)
        {
            const int tid = omp_get_thread_num();
            const size_t a = n * size_t(tid) / nt, b = n * size_t(tid + 1) / nt;
            size_t *h = hist.data() + size_t(tid) * NB;
            std::fill(h, h + NB, size_t(0));
            for (size_t p = a; p < b; ++p) ++h[(ks[p] >> shift) & (NB - 1)];
#pragma omp barrier
#pragma omp single
            {
                size_t run = 0;
                for (int d = 0; d < NB; ++d)
                    for (int t = 0; t < nt; ++t) {
                        size_t c = hist[size_t(t) * NB + d];
                        hist[size_t(t) * NB + d] = run;
                        run += c;
                    }
            }
            for (size_t p = a; p < b; ++p) {
                size_t q = h[(ks[p] >> shift) & (NB - 1)]++;
                kd[q] = ks[p];
                id[q] = is[p];
            }
        }
        keys.swap(k2);
        idx.swap(i2);
    }
}

}  // namespace

sa_status sa_build_levels(sa_tensor *t, const int32_t *coords, const float *vals)
{
    const int order = t->order;
    const int64_t nnz = t->nnz;
    int bits[SA_MAX_ORDER], shift[SA_MAX_ORDER];
    int total = 0;
    for (int d = 0; d < order; ++d) total += (bits[d] = bits_for(t->dims[d]));
    if (total > 64) return SA_E_UNSUPPORTED;
    for (int d = 0, s = total; d < order; ++d) { s -= bits[d]; shift[d] = s; }

    std::unique_ptr<uint64_t[]> keys;
    std::unique_ptr<uint32_t[]> idx;
    try {
        keys.reset(new uint64_t[size_t(nnz)]);
        idx.reset(new uint32_t[size_t(nnz)]);
    } catch (...) { return SA_E_ALLOC; }

    int bad = 0;
#pragma omp parallel for reduction(| : bad) schedule(static)
    for (int64_t p = 0; p < nnz; ++p) {
        uint64_t k = 0;
        for (int d = 0; d < order; ++d) {
            const int64_t c = coords[p * order + d];
            if (c < 0 || c >= t->dims[d]) bad |= 1;
            k |= uint64_t(uint32_t(c)) << shift[d];
        }
        keys[size_t(p)] = k;
        idx[size_t(p)] = uint32_t(p);
    }
    if (bad) return SA_E_COORD_RANGE;

    try { radix_sort(keys, idx, size_t(nnz), total); } catch (...) { return SA_E_ALLOC; }

    int dup = 0;
#pragma omp parallel for reduction(| : dup) schedule(static)
    for (int64_t p = 1; p < nnz; ++p)
        if (keys[size_t(p)] == keys[size_t(p - 1)]) dup |= 1;
    if (dup) return SA_E_COORD_DUP;

    try {
        t->vals.resize(size_t(nnz));
#pragma omp parallel for schedule(static)
        for (int64_t p = 0; p < nnz; ++p) t->vals[size_t(p)] = vals[idx[size_t(p)]];
        idx.reset();

        const int last = order - 1;
        auto coord_of = [&](uint64_t k, int d) { return int32_t((k >> shift[d]) & ((uint64_t(1) << bits[d]) - 1)); };

        if (t->fmt == SA_FMT_CSR) {
            const int64_t I = t->dims[0];
            t->count[0] = I;
            t->count[1] = nnz;
            t->pos[1].resize(size_t(I) + 1);
            t->crd[1].resize(size_t(nnz));
            // pos[r] = first entry of row r or of a later one: entry p sets it for the rows above the row of p - 1
#pragma omp parallel for schedule(static)
            for (int64_t p = 0; p <= nnz; ++p) {
                const int64_t row = p < nnz ? coord_of(keys[size_t(p)], 0) : I;
                for (int64_t r = p > 0 ? int64_t(coord_of(keys[size_t(p - 1)], 0)) + 1 : 0; r <= row; ++r) t->pos[1][size_t(r)] = p;
                if (p < nnz) t->crd[1][size_t(p)] = coord_of(keys[size_t(p)], 1);
            }
        } else {
            // prefix of level l = key >> shift[l]; a new node opens at every level >= the first
            // level whose prefix differs from the previous entry's
            auto first_new_level = [&](int64_t p) {
                if (p == 0) return 0;
                const uint64_t diff = keys[size_t(p)] ^ keys[size_t(p - 1)];
                int l = 0;
                while (l < last && (diff >> shift[l]) == 0) ++l;
                return l;
            };
            // two passes over fixed shares of the entries: how many nodes open in a share, then where they go
            const int nt = std::max(1, omp_get_max_threads());
            std::vector<int64_t> opened(size_t(nt + 1) * SA_MAX_ORDER, 0);
            auto share = [&](int w) { return nnz * w / nt; };
#pragma omp parallel for schedule(static) num_threads(nt)
            for (int w = 0; w < nt; ++w) {
                int64_t cnt[SA_MAX_ORDER] = {0, 0, 0, 0};
                for (int64_t p = share(w); p < share(w + 1); ++p)
                    for (int l = first_new_level(p); l < last; ++l) ++cnt[l];
                for (int l = 0; l < last; ++l) opened[size_t(w + 1) * SA_MAX_ORDER + size_t(l)] = cnt[l];
            }
            for (int w = 0; w < nt; ++w)
                for (int l = 0; l < last; ++l) opened[size_t(w + 1) * SA_MAX_ORDER + size_t(l)] += opened[size_t(w) * SA_MAX_ORDER + size_t(l)];
            for (int l = 0; l <= last; ++l) {
                t->count[l] = l == last ? nnz : opened[size_t(nt) * SA_MAX_ORDER + size_t(l)];
                t->crd[l].resize(size_t(t->count[l]));
                if (l < last) t->pos[l + 1].resize(size_t(t->count[l]) + 1);
            }
            for (int l = 0; l < last; ++l) t->pos[l + 1][size_t(t->count[l])] = t->count[l + 1];
            t->pos[0] = {0, t->count[0]};
#pragma omp parallel for schedule(static) num_threads(nt)
            for (int w = 0; w < nt; ++w) {
                int64_t at[SA_MAX_ORDER] = {0, 0, 0, 0};
                for (int l = 0; l < last; ++l) at[l] = opened[size_t(w) * SA_MAX_ORDER + size_t(l)];
                for (int64_t p = share(w); p < share(w + 1); ++p) {
                    const uint64_t k = keys[size_t(p)];
                    const int first = first_new_level(p);
                    for (int l = last - 1; l >= first; --l) t->pos[l + 1][size_t(at[l])] = l + 1 == last ? p : at[l + 1];
                    for (int l = first; l < last; ++l) t->crd[l][size_t(at[l]++)] = coord_of(k, l);
                    t->crd[last][size_t(p)] = coord_of(k, last);
                }
            }
        }
    } catch (...) { return SA_E_ALLOC; }
    return SA_OK;
}

// ------------------------------------------------------------------------------ work lists

namespace {

sa_item empty_item()
{
    sa_item it;
    it.out_row = 0; it.row_end = 0; it.f0 = 0; it.f1 = 0; it.p0 = 0; it.p1 = 0; it.dest = -1; it.pad = 0;
    return it;
}

struct group_rec { int64_t len; std::vector<sa_item> items; };

// Chunk of nonzeros one CTA reduces into a single tile: at least min_chunk, and large enough that
// a slice is cut into at most max_parts partial tiles.
int64_t chunk_for(int64_t n, int64_t min_chunk, int64_t max_parts)
{
    int64_t c = (n + max_parts - 1) / max_parts;
    c = ((c + min_chunk - 1) / min_chunk) * min_chunk;
    return std::max(c, min_chunk);
}

void append_empty_slices(sa_tensor *t, sa_worklist &wl)
{
    const int64_t I = t->dims[0];
    size_t s = 0;
    for (int64_t i = 0; i < I; ++i) {
        if (s < t->crd[0].size() && t->crd[0][s] == i) { ++s; continue; }
        wl.fix.push_back(sa_fix{int32_t(i), 0, 0, 0});
    }
}

// Items by decreasing number of nonzeros, items of equal length in the order they have.  Lengths are at most 4096 in all lists,
// so they are counted: building a 500 K nonzero CSR tensor takes 4.5 ms, with a comparison sort 5.6.
void longest_first(std::vector<sa_item> &items)
{
    auto len = [](const sa_item &x) { return size_t(x.p1 - x.p0); };
    size_t top = 0;
    for (const sa_item &x : items) top = std::max(top, len(x));
    std::vector<size_t> at(top + 2, 0);                  // at[top - len]: where the next item of that length goes
    for (const sa_item &x : items) ++at[top - len(x) + 1];
    for (size_t k = 1; k < at.size(); ++k) at[k] += at[k - 1];
    std::vector<sa_item> sorted(items.size());
    for (const sa_item &x : items) sorted[at[top - len(x)]++] = x;
    items.swap(sorted);
}

// Chunk into which a slice of n > unit nonzeros is cut (192 partial tiles per slice at most), and the partial tiles of all slices.
int64_t ttm3_chunk(int64_t n, int64_t unit) { return chunk_for(n, 4 * unit, 192); }
int64_t ttm3_slots(const std::vector<int64_t> &len, int64_t unit)
{
    int64_t slots = 0;
    for (const int64_t n : len) {
        const int64_t ng = n > unit ? (n - 1) / ttm3_chunk(n, unit) + 1 : 1;
        if (ng > 1) slots += ng;
    }
    return slots;
}

// Small slices per task: several only when there are enough of them to fill the machine (a few thousand warps) anyway.
int64_t ttm3_task_units(int64_t n_small) { return std::min<int64_t>(16, std::max<int64_t>(1, n_small / 4096)); }

// Time of the order-3 kernel on slices of the given lengths with units of `unit` nonzeros, in nonzeros of one warp: the thread
// blocks of the list in launch order on the `resident` slots of the machine, each for as long as its longest warp plus a fixed
// cost; blocks also run faster while fewer are resident, so their sum over the slots has a share.  A partial tile and the
// launch that adds them cost something too.  short_len[n]: slices of n nonzeros; long_len: the slices above 2048.
// `fibers` per nonzero: a nonzero takes the longer the more of them end a fiber, and the fixed costs count the less.
// The constants are fitted to 32 tensors of 0.15 to 7 M nonzeros (equal and Zipf slices, mean fibers of 1.5 to 20) at up to six
// combinations of ranks, each timed with seven unit sizes: the one that ttm3_unit takes is 1.3 % slower than the fastest in the
// mean, 16 % at most.
constexpr int64_t TTM3_UNITS[] = {2048, 1536, 1280, 1024, 896, 768, 640, 512, 384, 256};
double ttm3_time(const std::vector<int64_t> &short_len, const std::vector<int64_t> &long_len, double fibers, int64_t unit, int64_t slots, int64_t resident)
{
    constexpr double MAKESPAN_SHARE = 0.8;
    const double weight = 1.25 / (1 + 2 * fibers);                 // 1 for fibers of eight nonzeros
    const int64_t BLOCK_COST = int64_t(65 * weight), UNIT_COST = int64_t(32 * weight);      // UNIT_COST: each further unit of a task
    const double TILE_COST = 0.06 * weight, FIX_COST = 100 * weight;
    struct run_rec { int64_t cost, count; };
    std::vector<run_rec> blocks;
    auto cut = [&](int64_t n, int64_t count) {                    // the blocks of `count` slices of n > unit nonzeros
        const int64_t chunk = ttm3_chunk(n, unit), full = (n - 1) / chunk, rest = n - full * chunk;
        if (full > 0) blocks.push_back(run_rec{chunk / SA_TTM3_WARPS + BLOCK_COST, full * count});
        blocks.push_back(run_rec{(rest + SA_TTM3_WARPS - 1) / SA_TTM3_WARPS + BLOCK_COST, count});
    };
    for (const int64_t n : long_len) cut(n, 1);
    int64_t n_small = 0;
    for (int64_t n = int64_t(short_len.size()) - 1; n > 0; --n) {
        if (short_len[size_t(n)] == 0) continue;
        if (n > unit) cut(n, short_len[size_t(n)]);
        else n_small += short_len[size_t(n)];
    }
    std::sort(blocks.begin(), blocks.end(), [](const run_rec &x, const run_rec &y) { return x.cost > y.cost; });
    const int64_t max_units = ttm3_task_units(n_small);
    int64_t fill = 0, sum = 0, cnt = 0;                            // tasks in the last block; nonzeros and units of the open task
    auto emit = [&](int64_t nonzeros, int64_t units, int64_t tasks) {
        const int64_t more = std::min<int64_t>(tasks, fill > 0 ? SA_TTM3_WARPS - fill : 0);
        fill = (fill + tasks) % SA_TTM3_WARPS;
        tasks -= more;
        if (tasks > 0)
            blocks.push_back(run_rec{nonzeros + (units - 1) * UNIT_COST + BLOCK_COST, (tasks + SA_TTM3_WARPS - 1) / SA_TTM3_WARPS});
    };
    for (int64_t n = unit; n > 0; --n) {
        int64_t count = short_len[size_t(n)];
        if (count > 0 && cnt > 0) {
            const int64_t more = std::min(count, std::min(max_units - cnt, (unit - sum) / n));
            sum += more * n;
            cnt += more;
            count -= more;
            if (count > 0) { emit(sum, cnt, 1); sum = cnt = 0; }
        }
        if (count > 0) {
            const int64_t k = std::min(max_units, unit / n);
            if (count >= k) emit(k * n, k, count / k);
            cnt = count % k;
            sum = cnt * n;
        }
    }
    if (cnt > 0) emit(sum, cnt, 1);
    double total = 0;
    int64_t n_blocks = 0;
    for (const run_rec &x : blocks) { total += double(x.cost) * double(x.count); n_blocks += x.count; }
    const double even = total / double(resident);
    double last = even;
    if (n_blocks <= 16 * resident) {                               // more than 16 rounds: any order fills the machine
        std::vector<int64_t> busy(size_t(std::min<int64_t>(n_blocks, resident)), 0);    // a heap with the earliest free slot on top
        int64_t end = 0;
        for (const run_rec &x : blocks)
            for (int64_t c = 0; c < x.count; ++c) {
                std::pop_heap(busy.begin(), busy.end(), std::greater<int64_t>());
                busy.back() += x.cost;
                end = std::max(end, busy.back());
                std::push_heap(busy.begin(), busy.end(), std::greater<int64_t>());
            }
        last = double(end);
    }
    return MAKESPAN_SHARE * last + (1 - MAKESPAN_SHARE) * even + (slots > 0 ? FIX_COST + TILE_COST * double(slots) : 0.0);
}

// Nonzeros per unit: the largest of TTM3_UNITS within 1 % of the shortest estimated time, among those that need at most
// 1024 partial tiles (what sa_run_ttm3_static_scratch has room for at the largest ranks) or as many as units of 2048 need.
// From two units of 2048 per warp slot of the machine on it is 2048: balance is then not what the time goes to.
// L = M = 32, us, units of 2048 / what the rule takes: 300 slices of 1000 nonzeros 50 / 21, 1000 x 1100 35 / 29, 3000 x 400
// 45 / 45 (512 or more; 52 with 256), 50 x 40 000 60 / 43, 30 x 133 000 75 / 75 (83 with 832).
// *six_blocks: the 16 x 16 kernel compiled for six blocks per SM (fewer registers, each block 1.3 times as long) is through
// sooner than the one for four; left alone for large tensors.  16 x 16, us, four / six blocks: 1000 slices of 2000 nonzeros
// 33 / 39, 10 x 120 000 23 / 25, 400 x 8000 47 / 55, 3000 x 400 34 / 27, 800 x 700 21 / 15, 3000 x 2000 159 / 139.
int64_t ttm3_unit(const std::vector<int64_t> &len, int64_t n_fibers, int *six_blocks)
{
    constexpr int64_t LARGEST = TTM3_UNITS[0];
    int64_t nnz = 0;
    for (const int64_t n : len) nnz += n;
    if (nnz >= LARGEST * 2 * SA_SMS * 16) return LARGEST;
    std::vector<int64_t> short_len(size_t(LARGEST) + 1, 0), long_len;
    for (const int64_t n : len)
        if (n > LARGEST) long_len.push_back(n);
        else ++short_len[size_t(n)];
    const int64_t most = std::max<int64_t>(1024, ttm3_slots(len, LARGEST));
    const double fibers = double(n_fibers) / double(std::max<int64_t>(1, nnz));
    constexpr int COUNT = int(std::size(TTM3_UNITS));
    double time[COUNT], best = 1e300;
    std::atomic<bool> failed{false};
#pragma omp parallel for schedule(dynamic, 1)
    for (int x = 0; x < COUNT; ++x) {
        try {
            const int64_t slots = ttm3_slots(len, TTM3_UNITS[x]);
            time[x] = slots > most ? 1e300 : ttm3_time(short_len, long_len, fibers, TTM3_UNITS[x], slots, 4 * SA_SMS);
        } catch (...) { failed = true; }
    }
    if (failed) throw std::bad_alloc();
    for (const double x : time) best = std::min(best, x);
    int x = 0;
    while (time[x] > 1.01 * best) ++x;
    *six_blocks = 1.3 * ttm3_time(short_len, long_len, fibers, TTM3_UNITS[x], ttm3_slots(len, TTM3_UNITS[x]), 6 * SA_SMS) < time[x];
    return TTM3_UNITS[x];
}

// Nonzeros per unit of the order-4 lists, which hold the large (i,j) subtrees only: 2048, less where `nnz` nonzeros, of which
// these are a part, would give fewer than 2048 units.  4.2 M nonzeros: 439 us with 2048, 484 us with 256.
int64_t ttm4_unit(int64_t nnz) { return std::min<int64_t>(2048, std::max<int64_t>(256, nnz / 2048 / 64 * 64)); }

// Order-3 CSF.  An item ("unit") is a piece [p0, p1) of one slice with the fibers [f0, f1) it touches (a
// fiber may be cut between two units, each adds its part).  Slices above SMALL_MAX nonzeros are cut into
// chunks; the SA_TTM3_WARPS warps of a thread block take equal pieces of a chunk and reduce their tiles on chip.
// Smaller slices are one unit each; a warp evaluates a task of up to ttm3_task_units such units, about
// SMALL_MAX nonzeros in total.  Inside a unit the warp's SA_STREAMS lane groups stream the parts given by
// sa_unit3_streams; stream_f0 holds the fiber in which each part starts.
// `n_slices` slices; slice s is output row row_of(s), owns the fibers [pos1[s], pos1[s + 1]) whose nonzeros are
// [pos2[f], pos2[f + 1]).  (Order 3: the slices of the tensor.  Order 4: the (i,j) subtrees, whose "fibers" are
// the (i,j,k) fibers; output row = index of the (i,j) fiber.)
template <typename RowOf, typename Skip>
void build_ttm3_lists(sa_worklist &wl, int64_t n_slices, RowOf row_of, Skip skip, const std::vector<int64_t> &pos1,
                      const std::vector<int64_t> &pos2, int64_t unit)
{
    const int64_t SMALL_MAX = unit;
    std::vector<sa_item> small;
    std::vector<group_rec> groups;
    for (int64_t s = 0; s < n_slices; ++s) {
        if (skip(s)) continue;                    // evaluated by another kernel
        const int64_t fa = pos1[size_t(s)], fb = pos1[size_t(s) + 1];
        const int64_t pa = pos2[size_t(fa)], pb = pos2[size_t(fb)];
        const int64_t n = pb - pa;
        const int32_t row = row_of(s);
        if (n <= SMALL_MAX) {
            sa_item it = empty_item();
            it.out_row = row; it.row_end = row + 1; it.pad = int32_t(s);
            it.f0 = int32_t(fa); it.f1 = int32_t(fb); it.p0 = int32_t(pa); it.p1 = int32_t(pb);
            small.push_back(it);
            continue;
        }
        const int64_t chunk = ttm3_chunk(n, unit);
        const int64_t ng = (n + chunk - 1) / chunk;
        int32_t slot0 = -1;
        if (ng > 1) {
            slot0 = int32_t(wl.n_slots);
            wl.fix.push_back(sa_fix{row, slot0, int32_t(ng), 0});
            wl.n_slots += ng;
        }
        for (int64_t g = 0; g < ng; ++g) {
            const int64_t ga = pa + g * chunk, gb = std::min(pb, ga + chunk);
            int64_t piece = (gb - ga + SA_TTM3_WARPS - 1) / SA_TTM3_WARPS;
            piece = (piece + 31) / 32 * 32;
            group_rec rec;
            rec.len = gb - ga;
            for (int w = 0; w < SA_TTM3_WARPS; ++w) {
                const int64_t qa = std::min(gb, ga + w * piece), qb = std::min(gb, qa + piece);
                if (qa >= qb) break;              // the remaining warps of this block have nothing to do
                sa_item it = empty_item();
                it.out_row = row; it.row_end = row + 1; it.pad = int32_t(s);
                it.dest = ng > 1 ? slot0 + int32_t(g) : -1;
                // fiber holding nonzero qa, and one past the fiber holding nonzero qb - 1
                const int64_t f0 = (std::upper_bound(pos2.begin() + fa, pos2.begin() + fb + 1, qa) - pos2.begin()) - 1;
                const int64_t f1 = (std::upper_bound(pos2.begin() + fa, pos2.begin() + fb + 1, qb - 1) - pos2.begin());
                it.f0 = int32_t(f0); it.f1 = int32_t(f1); it.p0 = int32_t(qa); it.p1 = int32_t(qb);
                rec.items.push_back(it);
            }
            groups.push_back(std::move(rec));
        }
    }
    std::stable_sort(groups.begin(), groups.end(), [](const group_rec &a, const group_rec &b) { return a.len > b.len; });
    longest_first(small);
    wl.n_group_ctas = int64_t(groups.size());
    wl.task_start.clear();
    for (auto &g : groups)
        for (int w = 0; w < SA_TTM3_WARPS; ++w) {
            wl.task_start.push_back(int32_t(wl.items.size()));
            if (size_t(w) < g.items.size()) wl.items.push_back(g.items[size_t(w)]);
        }
    const int64_t max_units = ttm3_task_units(int64_t(small.size()));
    for (size_t x = 0; x < small.size();) {
        wl.task_start.push_back(int32_t(wl.items.size()));
        int64_t sum = 0, cnt = 0;
        while (x < small.size() && cnt < max_units && (cnt == 0 || sum + (small[x].p1 - small[x].p0) <= SMALL_MAX)) {
            sum += small[x].p1 - small[x].p0;
            wl.items.push_back(small[x]);
            ++x; ++cnt;
        }
    }
    wl.task_start.push_back(int32_t(wl.items.size()));
    wl.stream_f0.resize(wl.items.size() * SA_STREAMS);
    for (size_t u = 0; u < wl.items.size(); ++u) {
        const sa_item &it = wl.items[u];
        int64_t lo[SA_STREAMS], hi[SA_STREAMS];
        sa_unit3_streams(it.p0, it.p1, lo, hi);
        for (int q = 0; q < SA_STREAMS; ++q) {
            int64_t f = it.f0;
            if (lo[q] < hi[q])
                f = (std::upper_bound(pos2.begin() + it.f0, pos2.begin() + it.f1 + 1, lo[q]) - pos2.begin()) - 1;
            wl.stream_f0[u * SA_STREAMS + size_t(q)] = int32_t(f);
        }
    }
}

void build_ttm3(sa_tensor *t, sa_worklist &wl)
{
    std::vector<int64_t> len(size_t(t->count[0]));
    for (int64_t s = 0; s < t->count[0]; ++s)
        len[size_t(s)] = t->pos[2][size_t(t->pos[1][size_t(s) + 1])] - t->pos[2][size_t(t->pos[1][size_t(s)])];
    build_ttm3_lists(wl, t->count[0], [&](int64_t s) { return t->crd[0][size_t(s)]; }, [](int64_t) { return false; }, t->pos[1],
                     t->pos[2], ttm3_unit(len, t->count[1], &wl.six_blocks));
    append_empty_slices(t, wl);
}


// A subtree (i,j) that the subtree kernel of pass 1 can take whole.
static bool subtree_is_small(const sa_tensor *t, int64_t f2)
{
    const auto &pos2 = t->pos[2], &pos3 = t->pos[3];
    const int64_t fa = pos2[size_t(f2)], fb = pos2[size_t(f2) + 1];
    return fb - fa <= SA_SUB_MAX_F3 && pos3[size_t(fb)] - pos3[size_t(fa)] <= SA_SUB_MAX_NNZ;
}

// Order-4 CSF, schedule SA_SCHED_FISSIONED: the chain is evaluated in two passes (see sa_ttm4_fis.cu).  Pass 1 runs the order-3 kernel with
// the large (i,j) subtrees as slices: `wl` gets the same lists as an order-3 tensor whose slices are those
// level-1 fibers (output row = fiber index); the small subtrees go to the subtree kernel's list.  Pass 2 contracts the per-fiber temporaries of each slice with rows of
// C: `wl2` holds one item per (piece of a slice, quarter of the 256 temporaries' columns); a slice with more
// than CHUNK_F fibers is cut into pieces whose partial tiles the fix-up kernel sums.
void build_ttm4_fissioned(sa_tensor *t, sa_worklist &wl, sa_worklist &wl2)
{
    build_ttm3_lists(wl, t->count[1], [](int64_t f) { return int32_t(f); }, [&](int64_t f) { return subtree_is_small(t, f); },
                     t->pos[2], t->pos[3], ttm4_unit(t->nnz));
    constexpr int64_t CHUNK_F = 512;
    const auto &pos1 = t->pos[1];
    std::vector<sa_item> items;
    for (int64_t s = 0; s < t->count[0]; ++s) {
        const int64_t fa = pos1[size_t(s)], fb = pos1[size_t(s) + 1];
        const int32_t row = t->crd[0][size_t(s)];
        const int64_t nc = (fb - fa + CHUNK_F - 1) / CHUNK_F;
        int32_t slot0 = -1;
        if (nc > 1) {
            slot0 = int32_t(wl2.n_slots);
            wl2.fix.push_back(sa_fix{row, slot0, int32_t(nc), 0});
            wl2.n_slots += nc;
        }
        for (int64_t c = 0; c < nc; ++c) {
            const int64_t f0 = fa + c * CHUNK_F, f1 = std::min(fb, fa + (c + 1) * CHUNK_F);
            // a piece of at most eight fibers (one tensor-core group) is one item that takes the four quarters in turn
            const int nq = f1 - f0 <= 8 ? 1 : 4;
            for (int qc = 0; qc < nq; ++qc) {
                sa_item it = empty_item();
                it.out_row = row; it.row_end = row + 1;
                it.f0 = int32_t(f0); it.f1 = int32_t(f1);
                it.p0 = it.f0; it.p1 = it.f1;          // size key: fibers
                it.dest = nc > 1 ? slot0 + int32_t(c) : -1;
                it.pad = nq == 1 ? 4 : qc;
                items.push_back(it);
            }
        }
    }
    // largest first: the tail of the launch is then made of the cheapest items
    std::stable_sort(items.begin(), items.end(), [](const sa_item &a, const sa_item &b) { return (a.f1 - a.f0) > (b.f1 - b.f0); });
    wl2.items = std::move(items);
    wl2.n_group_ctas = 0;
    append_empty_slices(t, wl2);
}

// Order 4, pass 1 on whole (i,j) subtrees: items are ranges of consecutive small subtrees (subtree_is_small) with
// at most SA_SUB_MAX_F3 level-2 fibers, SA_SUB_MAX_ROWS subtrees and about 512 nonzeros (f0/f1 = the fibers,
// p0/p1 = the nonzeros).  No subtree is cut, so there are no partial tiles; the large subtrees are in the main list.
void build_ttm4_subtrees(sa_tensor *t, sa_worklist &wl)
{
    const auto &pos2 = t->pos[2], &pos3 = t->pos[3];
    const int64_t F2 = t->count[1];
    constexpr int64_t TARGET_NNZ = 512;
    auto nnz_at = [&](int64_t f2) { return pos3[size_t(pos2[size_t(f2)])]; };
    std::vector<sa_item> items;
    int64_t r0 = 0;
    auto flush = [&](int64_t r1) {
        if (r1 > r0) {
            sa_item it = empty_item();
            it.out_row = int32_t(r0); it.row_end = int32_t(r1);
            it.f0 = int32_t(pos2[size_t(r0)]); it.f1 = int32_t(pos2[size_t(r1)]);
            it.p0 = int32_t(nnz_at(r0)); it.p1 = int32_t(nnz_at(r1));
            items.push_back(it);
        }
        r0 = r1;
    };
    for (int64_t r = 0; r < F2; ++r) {
        if (!subtree_is_small(t, r)) {
            flush(r);
            r0 = r + 1;
            continue;
        }
        if (r > r0 && (pos2[size_t(r) + 1] - pos2[size_t(r0)] > SA_SUB_MAX_F3 || r - r0 >= SA_SUB_MAX_ROWS ||
                       nnz_at(r + 1) - nnz_at(r0) > TARGET_NNZ))
            flush(r);
    }
    flush(F2);
    for (const sa_item &it : items) wl.nnz += it.p1 - it.p0;
    wl.items = std::move(items);
    wl.n_group_ctas = 0;
}

// Order-4 CSF (see sa_ttm4.cu).  The chain runs as one fused kernel over *pieces*: contiguous ranges of (i,j)
// subtrees holding about PIECE_NNZ nonzeros, one thread block each.  A piece is a run of *super-items* (at most
// SA_F4_POOL subtrees: what the block's pool of 16 x 16 temporaries holds), a super-item a run of *items* that
// the block's warps take one at a time:
//   kind 0: at most 32 consecutive subtrees, about an eighth of the super-item's nonzeros (the kernel evaluates
//           their level-2 fibers in batches of at most SA_F4_ROWS);   f0/f1 = fibers, p0/p1 = nonzeros
//   kind 1: up to 8 consecutive *large* subtrees (more than SA_SUB_MAX_NNZ nonzeros), whose temporaries the
//           order-3 kernel has written beforehand; f0 = index of the first one among the large subtrees.
// Nothing is cut at a slice boundary: the block follows the slices through pos[1] while it consumes the
// temporaries.  A slice that lies in several pieces gets one partial tile per piece (consecutive slots) and a
// fix-up entry.  `wl` (main list): the order-3 lists over the large subtrees, output row = index among them.
static bool subtree_is_large(const sa_tensor *t, int64_t f2)
{
    const auto &pos2 = t->pos[2], &pos3 = t->pos[3];
    return pos3[size_t(pos2[size_t(f2) + 1])] - pos3[size_t(pos2[size_t(f2)])] > SA_SUB_MAX_NNZ;
}

void build_ttm4(sa_tensor *t, sa_worklist &wl, sa_worklist &wl_items, sa_worklist &wl_fix)
{
    const auto &pos1 = t->pos[1], &pos2 = t->pos[2], &pos3 = t->pos[3];
    const int64_t F2 = t->count[1], S = t->count[0];
    std::vector<int32_t> large_ord(size_t(F2), -1);
    int32_t n_large = 0;
    for (int64_t r = 0; r < F2; ++r)
        if (subtree_is_large(t, r)) large_ord[size_t(r)] = n_large++;
    t->f4_n_large = n_large;
    build_ttm3_lists(wl, F2, [&](int64_t r) { return large_ord[size_t(r)]; }, [&](int64_t r) { return large_ord[size_t(r)] < 0; },
                     pos2, pos3, ttm4_unit(t->nnz));
    wl.nnz = 0;
    for (const sa_item &it : wl.items) wl.nnz += it.p1 - it.p0;

    constexpr int64_t PIECE_NNZ = 16384, LARGE_WEIGHT = 64;
    auto nnz_at = [&](int64_t r) { return pos3[size_t(pos2[size_t(r)])]; };
    std::vector<sa_item> &items = wl_items.items;
    std::vector<int32_t> &supers = t->f4_supers, &pieces = t->f4_pieces;
    auto push_item = [&](int64_t r0, int64_t r1, int kind) {
        sa_item it = empty_item();
        it.out_row = int32_t(r0); it.row_end = int32_t(r1); it.pad = kind;
        if (kind == 0) {
            it.f0 = int32_t(pos2[size_t(r0)]); it.f1 = int32_t(pos2[size_t(r1)]);
            it.p0 = int32_t(nnz_at(r0)); it.p1 = int32_t(nnz_at(r1));
        } else {
            it.f0 = large_ord[size_t(r0)]; it.f1 = it.f0 + int32_t(r1 - r0);
        }
        items.push_back(it);
    };
    // One super-item = the subtrees [r0, r1), r1 - r0 <= SA_F4_POOL.  Its small subtrees are cut into at most SA_F4_WARPS
    // nonzero-balanced runs (one per warp of the block); a run also ends at a large subtree and after 32 subtrees.
    auto push_super = [&](int64_t r0, int64_t r1) {
        int64_t small_nnz = 0;
        for (int64_t r = r0; r < r1; ++r)
            if (large_ord[size_t(r)] < 0) small_nnz += nnz_at(r + 1) - nnz_at(r);
        const int64_t target = (small_nnz + SA_F4_WARPS - 1) / SA_F4_WARPS;
        const int32_t item0 = int32_t(items.size());
        int64_t run0 = r0, run_nnz = 0;
        int run_kind = -1;
        for (int64_t r = r0; r < r1; ++r) {
            const int kind = large_ord[size_t(r)] >= 0 ? 1 : 0;
            const bool full = run_kind >= 0 && (kind != run_kind || (kind == 1 ? r - run0 >= 8 : (run_nnz >= target || r - run0 >= 32)));
            if (full) { push_item(run0, r, run_kind); run_kind = -1; }
            if (run_kind < 0) { run_kind = kind; run0 = r; run_nnz = 0; }
            if (kind == 0) run_nnz += nnz_at(r + 1) - nnz_at(r);
        }
        if (run_kind >= 0) push_item(run0, r1, run_kind);
        supers.push_back(item0); supers.push_back(int32_t(items.size()));
        supers.push_back(int32_t(r0)); supers.push_back(int32_t(r1));
    };
    // slice that holds subtree r (r < F2)
    auto slice_of = [&](int64_t r) { return int64_t(std::upper_bound(pos1.begin(), pos1.end(), r) - pos1.begin()) - 1; };
    auto push_piece = [&](int64_t r0, int64_t r1) {
        const int32_t sup0 = int32_t(supers.size() / 4);
        for (int64_t r = r0; r < r1; r += SA_F4_POOL) push_super(r, std::min<int64_t>(r1, r + SA_F4_POOL));
        pieces.push_back(sup0); pieces.push_back(int32_t(supers.size() / 4));
        pieces.push_back(int32_t(slice_of(r0))); pieces.push_back(int32_t(slice_of(r1 - 1)));
        pieces.push_back(-1); pieces.push_back(-1);       // destinations of the first / last slice: set below
        pieces.push_back(int32_t(r0)); pieces.push_back(int32_t(r1));
    };
    {
        int64_t piece_r0 = 0, piece_w = 0;
        for (int64_t r = 0; r < F2; ++r) {
            if (piece_w >= PIECE_NNZ) { push_piece(piece_r0, r); piece_r0 = r; piece_w = 0; }
            piece_w += large_ord[size_t(r)] >= 0 ? LARGE_WEIGHT : nnz_at(r + 1) - nnz_at(r);
        }
        if (F2 > piece_r0) push_piece(piece_r0, F2);
    }
    wl_items.n_group_ctas = 0;
    // partial tiles: a slice that lies in more than one piece gets one slot per piece
    std::vector<int32_t> slice_slots(size_t(S), 0), slice_slot0(size_t(S), -1);
    const size_t n_pieces = pieces.size() / 8;
    for (size_t p = 0; p < n_pieces; ++p)
        for (int64_t s = pieces[8 * p + 2]; s <= pieces[8 * p + 3]; ++s) slice_slots[size_t(s)]++;
    for (int64_t s = 0; s < S; ++s)
        if (slice_slots[size_t(s)] > 1) {
            slice_slot0[size_t(s)] = int32_t(wl_fix.n_slots);
            wl_fix.fix.push_back(sa_fix{t->crd[0][size_t(s)], int32_t(wl_fix.n_slots), slice_slots[size_t(s)], 0});
            wl_fix.n_slots += slice_slots[size_t(s)];
        }
    std::vector<int32_t> next_slot(slice_slot0);
    for (size_t p = 0; p < n_pieces; ++p) {
        const int64_t sa = pieces[8 * p + 2], sb = pieces[8 * p + 3];
        if (slice_slot0[size_t(sa)] >= 0) pieces[8 * p + 4] = next_slot[size_t(sa)]++;
        if (sb != sa) { if (slice_slot0[size_t(sb)] >= 0) pieces[8 * p + 5] = next_slot[size_t(sb)]++; }
        else pieces[8 * p + 5] = pieces[8 * p + 4];
    }
    append_empty_slices(t, wl_fix);
}

// Rows of a sparse matrix given by its pos array: row ranges of about target_nnz nonzeros (at most max_rows rows); rows longer than
// long_thresh are cut into pieces of `piece` nonzeros whose partial rows the fix-up kernel sums.
// equal_parts: the pieces of a row have equal lengths, `piece` at most, and the list starts with the longest pieces.
// quarter_rows: a range item also records the rows that hold its nonzeros p0 + q ceil((p1 - p0) / 4), q = 1, 2, 3
// (fields f0, f1, pad), for kernels whose lane groups take equal counts of nonzeros rather than of rows.
void build_rows(const std::vector<int64_t> &pos, int64_t I, sa_worklist &wl, int64_t target_nnz, int64_t max_rows,
                int64_t long_thresh, int64_t piece, bool quarter_rows = false, bool equal_parts = false)
{
    std::vector<sa_item> longs, ranges;
    int64_t r0 = 0;
    auto flush = [&](int64_t r1) {
        if (r1 > r0) {
            sa_item it = empty_item();
            it.out_row = int32_t(r0); it.row_end = int32_t(r1);
            it.p0 = int32_t(pos[size_t(r0)]); it.p1 = int32_t(pos[size_t(r1)]);
            if (quarter_rows) {
                const int64_t share = (int64_t(it.p1) - it.p0 + 3) / 4;
                int32_t rows[3];
                for (int q = 1; q < 4; ++q) {
                    const int64_t at = std::min<int64_t>(int64_t(it.p0) + q * share, it.p1);
                    // the last row starting at or before `at`, inside the item
                    int64_t r = (std::upper_bound(pos.begin() + r0, pos.begin() + r1 + 1, at) - pos.begin()) - 1;
                    rows[q - 1] = int32_t(std::min<int64_t>(std::max<int64_t>(r, r0), r1 - 1));
                }
                it.f0 = rows[0]; it.f1 = rows[1]; it.pad = rows[2];
            }
            ranges.push_back(it);
        }
        r0 = r1;
    };
    for (int64_t r = 0; r < I; ++r) {
        const int64_t a = pos[size_t(r)], b = pos[size_t(r) + 1];
        if (b - a > long_thresh) {
            flush(r);
            const int64_t np = (b - a + piece - 1) / piece, part = equal_parts ? (b - a + np - 1) / np : piece;
            const int32_t slot0 = int32_t(wl.n_slots);
            wl.fix.push_back(sa_fix{int32_t(r), slot0, int32_t(np), 0});
            wl.n_slots += np;
            for (int64_t q = 0; q < np; ++q) {
                sa_item it = empty_item();
                it.out_row = int32_t(r); it.row_end = int32_t(r + 1);
                it.p0 = int32_t(std::min(b, a + q * part)); it.p1 = int32_t(std::min(b, a + (q + 1) * part));
                it.dest = slot0 + int32_t(q);
                longs.push_back(it);
            }
            r0 = r + 1;
            continue;
        }
        if (pos[size_t(r) + 1] - pos[size_t(r0)] > target_nnz && r > r0) flush(r);
        if (r + 1 - r0 >= max_rows) flush(r + 1);
    }
    flush(I);
    // longest first: the tail of the launch is then made of the cheapest items
    longest_first(ranges);
    if (equal_parts) longest_first(longs);
    wl.n_group_ctas = 0;
    wl.items = std::move(longs);
    wl.items.insert(wl.items.end(), ranges.begin(), ranges.end());
}

// CSR, row kernel of the left orders (spmm_gemm_left_kernel): the most nonzeros a row may have without being cut.  Cutting a
// row costs a product of its part with D (row_cost nonzeros' time) per piece, and the gathers of the pieces run at the rate of
// HBM, which is what cut_warps warps reach; so do those of whole rows unless columns are used several times (nnz > 2 J): then
// all warps walk through the columns together and find C in L2.  Cutting pays where few or very unequal rows leave warps
// idle.  Time in nonzeros of one warp: the kernel's warps take items in turn, longest first, so the first one of each round
// counts.  Rows stay whole if no cut is 2 % faster, else the largest limit within 2 % of the shortest time is taken.
// L = 256, M = 64, us, rows of up to 4096 whole / cut at nnz / 18944 nonzeros / by this rule: 2000 rows of 600 nonzeros 130 /
// 200 / 130 (kernel 3: 211 / 417 / 211), 3000 of 1000 215 / 430 / 215, 500 of 1000 231 / 103 / 94, 500 of 3000 555 / 242 / 182,
// 3 M nonzeros on 100 K rows, Zipf(1.2) 1230 / 650 / 680.
int64_t left_row_limit(const std::vector<int64_t> &pos, int64_t I, int64_t J, int64_t target, int64_t row_cost, int64_t cut_warps)
{
    constexpr int64_t LIMITS[] = {4096, 2048, 1024, 512, 256, 128, 64, 32}, WARPS = SA_SMS * 24, FIX_COST = 40;   // FIX_COST: the launch that adds the pieces
    std::vector<int64_t> count(size_t(LIMITS[0]) + 1, 0), over;
    for (int64_t r = 0; r < I; ++r) {
        const int64_t n = pos[size_t(r) + 1] - pos[size_t(r)];
        if (n > LIMITS[0]) over.push_back(n);
        else ++count[size_t(n)];
    }
    const int64_t nnz = pos[size_t(I)];
    double best = 1e300, time[std::size(LIMITS)];
    for (size_t x = 0; x < std::size(LIMITS); ++x) {
        const int64_t limit = LIMITS[x], piece = std::min<int64_t>(limit, 2048);
        std::vector<int64_t> len(count.begin(), count.begin() + limit + 1);      // items by length (short rows as if one each)
        bool cut = false;
        auto add = [&](int64_t n, int64_t rows) {
            cut = true;
            const int64_t parts = (n + piece - 1) / piece;
            len[size_t((n + parts - 1) / parts)] += rows * parts;
        };
        for (int64_t n = limit + 1; n <= LIMITS[0]; ++n)
            if (count[size_t(n)] > 0) add(n, count[size_t(n)]);
        for (const int64_t n : over) add(n, 1);
        double first = 0, short_nnz = 0, short_rows = 0;
        int64_t at = 0;                                                         // items longer than `target` so far
        for (int64_t n = limit; n >= 0; --n) {
            const int64_t c = len[size_t(n)];
            if (n <= target) {
                short_nnz += double(c * n);
                short_rows += double(c);
                continue;
            }
            first += double((at + c + WARPS - 1) / WARPS - (at + WARPS - 1) / WARPS) * double(n + row_cost);
            at += c;
        }
        // ranges of short rows: `target` nonzeros or 16 rows; they begin in the last round of the long items
        const double rows_each = std::min(16.0, std::max(1.0, double(target) * short_rows / std::max(1.0, short_nnz)));
        const double each = std::max(1.0, rows_each * (short_nnz / std::max(1.0, short_rows) + double(row_cost)));
        const double ranges = short_rows / rows_each, room = double((at + WARPS - 1) / WARPS * WARPS - at);
        time[x] = std::max(first + std::max(0.0, ranges - room) / WARPS * each, short_rows > 0 ? each : 0.0) + (cut ? FIX_COST : 0);
        best = std::min(best, time[x]);
    }
    const double from_hbm = double(nnz) / double(cut_warps);
    if (std::max(time[0], nnz > 2 * J ? 0.0 : from_hbm) <= 1.02 * std::max(best, from_hbm)) return LIMITS[0];
    size_t x = 1;
    while (time[x] > 1.02 * best) ++x;
    return LIMITS[x];
}

// CSR, kernel 1 (fused SDDMM -> SpMM): an item is what one group of eight lanes walks, a range of whole short rows or a
// piece of a long row with a partial row for the fix-up kernel.
//   Size: `target` nonzeros, at most 256, less where the tensor would not give every group of a full machine
//     (64 groups per SM) two items, at least 16: a group needs about a microsecond per four nonzeros, and on a small tensor
//     that chain is the whole run time (60 k nonzeros, rows of up to 1500: 28 us; with a warp per item of up to 1024
//     nonzeros 78 us).  A row counts as long above 64 nonzeros (1M x 1M, 30 M nonzeros: above 64 / 128 / 256 / 1024
//     1.01 / 1.03 / 1.05 / 1.09 ms).  Rows per range: 8, at least 4, by the same rule, since a
//     range of nearly empty rows is a chain of row loads and stores (whole call with the dense stage, 60 k nonzeros on 6 K
//     rows 24.6 us with 32 rows, 18.2 with 4; 3 M nonzeros on 1 M rows and columns, Zipf(1.2), K = L = 32 236 us with 32, 213
//     with 16, 200 with 8; K = 64, L = 32 309, 291, 278).
//   Order: D and E are gathered by column, and with J x (K + L) floats above L2 the order of the work decides what is
//     found there.  Rows above CUT_ROW nonzeros are therefore cut where their columns cross a multiple of COL_BLOCK (a piece
//     has at least MIN_PIECE nonzeros, since each costs a partial row) and the pieces are sorted by block: whatever runs at one
//     time then gathers from the same few blocks (32 K columns x (64 + 64) floats = 16 MB).  1M x 1M, 30 M nonzeros,
//     K = L = 64: 1.05 ms with blocks of 32 K or 64 K columns, 1.06 with 16 K.  Shorter rows stay whole: their pieces would be
//     mostly partial rows.  K = L = 64, us, cut / whole: rows of 100 nonzeros, 1 M columns 526 / 516, 200 K 382 / 311, 100 K
//     343 / 273; rows of 200, 1 M columns 329 / 345, 200 K 246 / 251.  Pieces of at least 16 instead of 32 nonzeros need up to
//     twice the workspace: rows of 300, 1 M columns 249 / 222, K = L = 128 687 / 699.
//     Inside a block the longest pieces come first, so that the four groups of a warp get pieces of like length.
void build_sddmm(const std::vector<int64_t> &pos, const std::vector<int32_t> &crd, int64_t I, sa_worklist &wl)
{
    constexpr int64_t COL_BLOCK = 32768, MIN_PIECE = 32, CUT_ROW = 128, MIN_REST = 16;
    const int64_t target = std::min<int64_t>(256, std::max<int64_t>(16, pos[size_t(I)] / (2 * SA_SMS * 64)));
    const int64_t long_row = std::min<int64_t>(std::max<int64_t>(target, 48), 64);
    const int64_t max_rows = std::min<int64_t>(8, std::max<int64_t>(4, I / (2 * SA_SMS * 64)));
    struct piece_rec { uint32_t key; sa_item it; };
    std::vector<piece_rec> pieces;
    std::vector<sa_item> ranges;
    int64_t r0 = 0;
    auto flush = [&](int64_t r1) {
        if (r1 > r0) {
            sa_item it = empty_item();
            it.out_row = int32_t(r0); it.row_end = int32_t(r1);
            it.p0 = int32_t(pos[size_t(r0)]); it.p1 = int32_t(pos[size_t(r1)]);
            ranges.push_back(it);
        }
        r0 = r1;
    };
    for (int64_t r = 0; r < I; ++r) {
        const int64_t a = pos[size_t(r)], b = pos[size_t(r) + 1];
        if (b - a > long_row) {
            flush(r);
            const size_t first = pieces.size();
            for (int64_t p = a; p < b;) {
                int64_t q = std::min(b, p + target);
                // the first block boundary after MIN_PIECE nonzeros, if there is one before q
                if (b - a > CUT_ROW && q - p > MIN_PIECE && crd[size_t(q) - 1] / COL_BLOCK != crd[size_t(p + MIN_PIECE) - 1] / COL_BLOCK) {
                    const int32_t edge = int32_t((crd[size_t(p + MIN_PIECE) - 1] / COL_BLOCK + 1) * COL_BLOCK);
                    q = std::lower_bound(crd.begin() + p + MIN_PIECE, crd.begin() + q, edge) - crd.begin();
                }
                if (b - q < MIN_REST) q = b;
                sa_item it = empty_item();
                it.out_row = int32_t(r); it.row_end = int32_t(r + 1);
                it.p0 = int32_t(p); it.p1 = int32_t(q);
                pieces.push_back(piece_rec{uint32_t(crd[size_t(p)] / COL_BLOCK), it});
                p = q;
            }
            const int64_t np = int64_t(pieces.size() - first);
            if (np > 1) {
                for (size_t x = first; x < pieces.size(); ++x) pieces[x].it.dest = int32_t(wl.n_slots + int64_t(x - first));
                wl.fix.push_back(sa_fix{int32_t(r), int32_t(wl.n_slots), int32_t(np), 0});
                wl.n_slots += np;
            }
            r0 = r + 1;
            continue;
        }
        if (pos[size_t(r) + 1] - pos[size_t(r0)] > target && r > r0) flush(r);
        if (r + 1 - r0 >= max_rows) flush(r + 1);
    }
    flush(I);
    std::sort(pieces.begin(), pieces.end(), [](const piece_rec &x, const piece_rec &y) {
        if (x.key != y.key) return x.key < y.key;
        const int32_t lx = x.it.p1 - x.it.p0, ly = y.it.p1 - y.it.p0;
        return lx != ly ? lx > ly : x.it.p0 < y.it.p0;
    });
    longest_first(ranges);
    wl.n_group_ctas = 0;
    wl.items.clear();
    wl.items.reserve(pieces.size() + ranges.size());
    for (const piece_rec &x : pieces) wl.items.push_back(x.it);
    wl.items.insert(wl.items.end(), ranges.begin(), ranges.end());
}

}  // namespace

void sa_build_worklists(sa_tensor *t)
{
    if (t->fmt == SA_FMT_CSF && t->order == 3) {
        build_ttm3(t, t->wl_main);
        // kernel 7 walks the tensor as a sparse matrix whose rows are the (i,j) fibers: 1024 nonzeros per warp, fewer where
        // that would not give every warp slot of a full machine four items
        build_rows(t->pos[2], t->count[1], t->wl_aux, std::min<int64_t>(1024, std::max<int64_t>(128, t->nnz / (4 * SA_SMS * 32) / 32 * 32)), 4096, 4096, 2048, true);
    }
    if (t->fmt == SA_FMT_CSF && t->order == 4) {
        build_ttm4(t, t->wl_main, t->wl_sub, t->wl_aux);
        build_ttm4_fissioned(t, t->wl4_main, t->wl4_aux);
        build_ttm4_subtrees(t, t->wl4_sub);
        t->wl4_main.nnz = t->nnz - t->wl4_sub.nnz;
    }
    if (t->fmt == SA_FMT_CSR) {
        // SpMM -> GEMM, the SpMM stage of the right orders (wl_aux) and the row kernel of the left ones (wl_sub, wl4_sub): about
        // 256 nonzeros per item, which one lane group or warp walks as a chain; fewer where the tensor would not give every
        // group of a full machine two items
        const std::vector<int64_t> &pos = t->pos[1];
        const int64_t I = t->dims[0], J = t->dims[1], target = std::min<int64_t>(256, std::max<int64_t>(32, t->nnz / (2 * SA_SMS * 64)));
        const int64_t wide = left_row_limit(pos, I, J, target, 50, 1200);      // 1 KB or more gathered per nonzero
        const int64_t narrow = left_row_limit(pos, I, J, target, 20, 2400);    // 512 bytes; no list of its own at the same limit
        std::atomic<bool> failed{false};
#pragma omp parallel for schedule(dynamic, 1)
        for (int list = 0; list < 4; ++list) {
            try {
                if (list == 0) build_sddmm(pos, t->crd[1], I, t->wl_main);
                if (list == 1) build_rows(pos, I, t->wl_aux, target, 16, 2 * target, target);
                if (list == 2) build_rows(pos, I, t->wl_sub, target, 16, wide, std::min<int64_t>(wide, 2048), false, true);
                if (list == 3 && narrow != wide) build_rows(pos, I, t->wl4_sub, target, 16, narrow, std::min<int64_t>(narrow, 2048), false, true);
            } catch (...) { failed = true; }
        }
        if (failed) throw std::bad_alloc();
    }
    for (sa_worklist *wl : {&t->wl_main, &t->wl_aux, &t->wl_sub, &t->wl4_main, &t->wl4_aux, &t->wl4_sub}) {
        std::stable_sort(wl->fix.begin(), wl->fix.end(), [](const sa_fix &x, const sa_fix &y) { return x.count > y.count; });
        wl->n_big_fix = std::find_if(wl->fix.begin(), wl->fix.end(), [](const sa_fix &x) { return x.count <= SA_BIG_FIX; }) - wl->fix.begin();
        wl->n_sum_fix = std::find_if(wl->fix.begin(), wl->fix.end(), [](const sa_fix &x) { return x.count == 0; }) - wl->fix.begin();
    }
}
