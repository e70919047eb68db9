// C ABI of libmate: argument checks, the plan object, and dispatch to the kernels.
#include <algorithm>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <exception>
#include <memory>
#include <new>

#include "mate_internal.h"

using mate::FwdUnit;
using mate::TileInfo;
using mate::kTile;
using mate::ViewPlan;

namespace {

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }
inline bool aligned16(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline int ceil_div(int a, int b) { return (a + b - 1) / b; }

// The entry points that make plans hold lists as long as their inputs: memory that is not to be had is a status
// there, never an exception across the C boundary.
template <typename F>
int no_throw(F &&f) {
    try {
        return f();
    } catch (const std::exception &) {
        return MATE_ERR_NOMEM;
    }
}

// Carves the plan's device arrays out of one allocation.
struct Carver {
    char *base;
    size_t off = 0;
    explicit Carver(char *b) : base(b) {}
    template <typename T>
    T *take(size_t n) {
        off = align_up(off, 256);
        T *p = base ? reinterpret_cast<T *>(base + off) : nullptr;
        off += n * sizeof(T);
        return p;
    }
};

// What is copied in before the plan kernel (prefix, global, head_view) and out behind it (segment offsets,
// numbers of valid positions, status) lies together, so that each is one copy.
struct PlanLayout {
    size_t total, in_off, in_bytes, out_off, out_bytes;
};
PlanLayout carve(mate_plan_t *pl, char *base) {
    Carver c(base);
    PlanLayout L;
    const size_t BN = (size_t)pl->B * pl->N;
    for (int v = 0; v < 2; ++v) {
        ViewPlan &vp = pl->view[v];
        vp.perm = c.take<int32_t>(BN);
        vp.inv_perm = c.take<int32_t>(BN);
        vp.seg_lo = c.take<int32_t>(BN);
        vp.seg_hi = c.take<int32_t>(BN);
        vp.cursor = c.take<int32_t>((size_t)pl->B * (vp.max_id + 2));
        vp.ident = c.take<int32_t>(pl->B);
    }
    L.in_off = c.off = align_up(c.off, 256);
    pl->prefix_dev = c.take<int32_t>(pl->B);
    pl->global_dev = c.take<int32_t>(pl->B);
    pl->head_view_dev = c.take<uint8_t>(pl->H);
    c.off = align_up(c.off, 256);
    pl->status_dev = c.take<int32_t>(4);  // in both: comes in as zeros
    L.in_bytes = c.off - L.in_off;
    L.out_off = c.off - 4 * sizeof(int32_t);
    pl->n_valid_dev = c.take<int32_t>(pl->B);
    for (int v = 0; v < 2; ++v) pl->view[v].seg_off = c.take<int32_t>((size_t)pl->B * (pl->view[v].max_id + 2));
    L.out_bytes = c.off - L.out_off;
    L.total = align_up(c.off, 256);
    return L;
}

// Column range of one table row (view position t) of one (example, view): its segment, clipped to the
// three adjacent buckets when the plan is bucketed.  The same arithmetic as step 4 of the plan kernel.
struct RowBounds {
    const int32_t *so;
    int S, P, radius;  // P: length of the global block (bucket origin; no range reaches in front of it)
    int mode = mate::kBoundsOwn, group = 1;
    // range of the positions of segment `id`, without the buckets
    int own_lo(int id) const {
        return std::max(mode == mate::kBoundsBefore ? so[id / group * group] : mode == mate::kBoundsAfter ? so[id + 1] : so[id], P);
    }
    int own_hi(int id) const {
        return mode == mate::kBoundsBefore ? so[id] : mode == mate::kBoundsAfter ? so[std::min((id / group + 1) * group, S - 1)] : so[id + 1];
    }
    // the three adjacent buckets of position t (never beyond 2^31: positions are below 2^30)
    int bucket_lo(int t) const { return (int)std::max<int64_t>(P + (int64_t)((t - P) / radius - 1) * radius, P); }
    int bucket_hi(int t) const { return (int)std::min<int64_t>(P + (int64_t)((t - P) / radius + 2) * radius, INT32_MAX); }
};

// ---------------------------------------------------------------------------- work-lists
// Work-lists of the tensor-core kernels, built on the host from the segment offsets: the rows of every
// (example, view) are cut into units (see FwdUnit), the same for all heads of the view, and listed by
// decreasing cost; the CTAs take them from the head of the list through a counter.
constexpr int kChunk = 32;

// Key ranges of the rows of one (example, view), by view position.
struct RowRanges {
    int P = 0, nv = 0;  // [0, P): rows of the global block; [P, nv): table rows with the keys [lo, hi) behind the block
    int64_t own = 0;    // pairs of table rows and the keys of their own ranges
    std::unique_ptr<int32_t[]> both;  // (not cleared: the segments fill what is read of it)
    int32_t *lo = nullptr, *hi = nullptr;
    std::vector<int32_t> starts;      // table rows whose lo differs from the one before (ascending)
    void begin(int t, int l) {
        if (starts.empty() || lo[t - 1] != l) starts.push_back(t);
    }
};

void fill_ranges(const mate_plan_t *pl, const int32_t *const (&seg_off_host)[2], int v, int b, RowRanges &rr) {
    const int S = pl->view[v].max_id + 2;
    const int32_t *so = seg_off_host[v] + (size_t)b * S;
    const RowBounds rb{so, S, std::min(pl->global[b], pl->n_valid[b]), pl->radius, pl->bounds_mode, pl->group};
    rr.P = rb.P;
    rr.nv = pl->n_valid[b];
    rr.both.reset(new int32_t[2 * (size_t)rr.nv + 1]);
    rr.lo = rr.both.get();
    rr.hi = rr.lo + rr.nv;
    rr.starts.clear();
    rr.starts.reserve(256);
    for (int id = 0; id + 1 < S; ++id) {
        const int t0 = std::max(so[id], rb.P), t1 = so[id + 1];
        if (t1 <= t0) continue;
        const int l = rb.own_lo(id), h = std::max(rb.own_hi(id), l);
        if (pl->radius <= 0) {
            rr.begin(t0, l);
            std::fill(rr.lo + t0, rr.lo + t1, l);
            std::fill(rr.hi + t0, rr.hi + t1, h);
            rr.own += (int64_t)(t1 - t0) * (h - l);
            continue;
        }
        for (int t = t0; t < t1;) {  // bucket by bucket
            const int end = (int)std::min<int64_t>(t1, rb.P + (int64_t)((t - rb.P) / pl->radius + 1) * pl->radius);
            const int lo = std::max(l, rb.bucket_lo(t)), hi = std::max(std::min(h, rb.bucket_hi(t)), lo);
            rr.begin(t, lo);
            std::fill(rr.lo + t, rr.lo + end, lo);
            std::fill(rr.hi + t, rr.hi + end, hi);
            rr.own += (int64_t)(end - t) * (hi - lo);
            t = end;
        }
    }
}

// Estimated clocks of the forward kernel (fitted to its per-unit times): a half alone on a tile; both
// halves on a tile together take 0.72 of the sum.  A unit costs its loads, set-up and epilogue; a part of a
// split unit also writes its partial result and, in the end, somebody combines them.
constexpr int kFullClk = 1800, kPartialClk = 900, kChunkClk = 350, kUnitClk = 3500, kPartClk = 3000;

struct Proto {
    FwdUnit u;
    int view;
    int tile0, n_tiles;  // estimated clocks of its tiles: tiles[tile0 ..] of the list
    int64_t cost;        // of the whole unit
};
struct ProtoList {
    std::vector<Proto> protos;
    std::vector<int32_t> tiles;
};

// Adds the estimated clocks of half h on every tile of its unit to clk (none where it skips the tile).
void half_tile_clks(const FwdUnit &u, int h, const RowRanges &rr, int32_t *clk) {
    const int nA = u.tiles_a(), n_tiles = nA + u.tiles_b(), rows = u.rows_of(h), r0 = u.row0_of(h);
    if (rows == 0) return;
    for (int i = 0; i < nA; ++i) {  // every row counts every column
        const int w = std::min(u.kA_end - u.kA0 - i * kTile, kTile);
        clk[i] = w == kTile ? kFullClk : kPartialClk + kChunkClk * ceil_div(w, kChunk);
    }
    for (int i = nA; i < n_tiles; ++i) {
        const TileInfo t = mate::tile_info(u, i, nA);
        int c0, c1;
        mate::half_cols(u.lo[h], u.hi[h], t, c0, c1);
        if (c1 <= c0) continue;
        const auto lo = [&](int r) { return r < rr.P ? 0 : rr.lo[r] - t.k0; };
        const auto hi = [&](int r) { return r < rr.P ? t.w : std::min(rr.hi[r] - t.k0, t.w); };
        if (t.w == kTile && (t.pre == kTile || (lo(r0 + rows - 1) <= t.pre && hi(r0) >= kTile))) {
            clk[i] = kFullClk;
            continue;
        }
        int chunks = ceil_div(t.pre, kChunk);
        for (int r = 0; t.is_b && r < rows; r += 32) {  // the warps of the half
            const int last = r0 + std::min(r + 32, rows) - 1;
            const int a = std::max(lo(r0 + r), 0), e = hi(last);
            int n = e > a ? ceil_div(e, kChunk) - a / kChunk : 0;
            if (t.pre > 0) n = ceil_div(t.pre, kChunk) + (e > t.pre ? ceil_div(e, kChunk) - std::max(a / kChunk, ceil_div(t.pre, kChunk)) : 0);
            chunks = std::max(chunks, n);
        }
        clk[i] = kPartialClk + kChunkClk * chunks;
    }
}

void add_proto(ProtoList &pl, const FwdUnit &u, int view, const RowRanges &rr) {
    Proto pr{u, view, (int)pl.tiles.size(), u.tiles_a() + u.tiles_b(), kUnitClk};
    pl.tiles.resize(pr.tile0 + 2 * pr.n_tiles, 0);
    int32_t *a = pl.tiles.data() + pr.tile0, *b = a + pr.n_tiles;
    half_tile_clks(u, 0, rr, a);
    half_tile_clks(u, 1, rr, b);
    for (int i = 0; i < pr.n_tiles; ++i) {
        a[i] = a[i] && b[i] ? (a[i] + b[i]) * 18 / 25 : std::max(a[i] + b[i], 100);
        pr.cost += a[i];
    }
    pl.tiles.resize(pr.tile0 + pr.n_tiles);
    pl.protos.push_back(pr);
}

// Longest first; the heads of a view repeat its units.
void sort_protos(ProtoList &pl) {
    std::vector<std::pair<int64_t, int>> order(pl.protos.size());  // (the records are moved once)
    for (size_t i = 0; i < order.size(); ++i) order[i] = {-pl.protos[i].cost, (int)i};
    std::sort(order.begin(), order.end());
    std::vector<Proto> sorted;
    sorted.reserve(order.size());
    for (const auto &o : order) sorted.push_back(pl.protos[o.second]);
    pl.protos.swap(sorted);
}
struct HeadLists {
    std::vector<int> heads[2];
    explicit HeadLists(const mate_plan_t *pl) {
        for (int h = 0; h < pl->H; ++h) heads[pl->head_view[h]].push_back(h);
    }
};

// Tiles that the halves of a unit visit.
int visits(const FwdUnit &u) {
    const int nA = u.tiles_a(), n_tiles = nA + u.tiles_b();
    int n = nA * ((u.rows_of(0) > 0) + (u.rows_of(1) > 0));
    for (int i = nA; i < n_tiles; ++i)
        for (int h = 0; h < 2; ++h) {
            int c0, c1;
            mate::half_cols(u.lo[h], u.hi[h], mate::tile_info(u, i, nA), c0, c1);
            n += u.rows_of(h) > 0 && c1 > c0;
        }
    return n;
}
constexpr int kMaxMerged = 3 * kTile;  // longest global block that goes in front of range B

// The unit of the rows [r0, r1) and [r1, r2) (the second half may be empty) with the global block in range A
// or, where the halves then visit fewer tiles, in front of range B.  Rows of the global block may stand in
// front of table rows in a half.
FwdUnit make_unit(const RowRanges &rr, int r0, int r1, int r2) {
    FwdUnit u{};
    const int n = (r1 - r0) | (r2 - r1) << 8;
    u.q0 = r0;
    u.rows = n;
    u.tB = kTile;
    u.parts = 1;
    u.ctr = -1;
    if (r2 <= rr.P) {  // global rows only
        u.kA_end = rr.nv;
        return u;
    }
    const int r[3] = {r0, r1, r2};
    for (int h = 0; h < 2; ++h) {
        if (r[h + 1] <= r[h]) continue;
        u.lo[h] = r[h] < rr.P ? rr.P : rr.lo[r[h]];  // lo and hi do not decrease along the table rows
        u.hi[h] = r[h] < rr.P ? rr.nv : rr.hi[r[h + 1] - 1];
    }
    u.kB0 = u.lo[0];
    u.kB_end = std::max(u.hi[0], u.hi[1]);
    FwdUnit m = u;
    m.rows = n | rr.P << 16;
    if (r0 < rr.P) return m;  // a mixed half masks row by row
    u.kA_end = rr.P;
    // When the second half's keys begin at most a tile behind the first half's, tiles of that width give each
    // half one tile of its own (short segments: the keys of a half are its own rows).
    const int step = u.lo[1] - u.lo[0];
    if (r2 > r1 && step > 0 && step <= kTile && u.hi[0] - u.lo[0] <= step && u.hi[1] - u.lo[1] <= step) u.tB = step;
    const bool may = rr.P > 0 && rr.P % kTile != 0 && rr.P < kMaxMerged;
    return may && visits(m) < visits(u) ? m : u;
}

// Units of one (example, view), for any head of the view.  Padding rows are left out.  `pairs`: two halves
// to a unit where they share most of their tiles.  `fill_up`: see below.
void add_units(const RowRanges &rr, int b, int view, bool pairs, bool fill_up, ProtoList &out) {
    const int P = rr.P, nv = rr.nv;
    const auto add = [&](int r0, int r1, int r2) {
        FwdUnit u = make_unit(rr, r0, r1, r2);
        u.b = b;
        add_proto(out, u, view, rr);
    };
    const auto tiles = [&](int cols) {  // of a half whose own keys are that many: with the global block in either place
        return std::min(ceil_div(P, kTile) + ceil_div(cols, kTile), P < kMaxMerged ? ceil_div(P + cols, kTile) : 1 << 28);
    };
    // The last half of the global block is filled up with table rows: these need no half of their own then (its
    // tiles, and about two more for the half itself), but the half masks its tiles row by row, about 0.3 of a
    // tile each.  Always for up to two tiles of positions; for longer examples only where all SMs have several
    // units to do (`fill_up`: the half is the longest of its example) and it saves more than it costs.
    std::vector<int> cuts(1, 0);
    while (cuts.back() + kTile <= P) cuts.push_back(cuts.back() + kTile);
    const int rem = P - cuts.back(), fill = std::min(kTile - rem, nv - P);
    if (rem > 0) {
        bool mix = fill > 0 && P < kMaxMerged;
        if (mix && nv > 2 * kTile) {
            const int own = rr.hi[P + fill - 1] - rr.lo[P];
            mix = fill_up && 0.3 * ceil_div(nv, kTile) < (tiles(own) + 2) * fill / (double)kTile;
        }
        cuts.push_back(mix ? P + fill : P);
    }
    const int n_global = (int)cuts.size() - 1;  // halves with rows of the global block
    // Halves of table rows: 128 rows, or fewer when ending where a segment begins saves tiles (a half that
    // reaches into the next long segment visits the tiles of both; one that ends with a short segment needs
    // one tile for its own keys instead of two).  Measure: tiles, and 1.5 for the half itself, per row.
    size_t next_start = 0;  // the first one behind `end`
    while (cuts.back() < nv) {
        const int q = cuts.back();
        int end = std::min(q + kTile, nv);
        if (end < nv || rr.lo[end - 1] != rr.lo[q]) {
            while (next_start < rr.starts.size() && rr.starts[next_start] <= end) ++next_start;
            const int cut = next_start > 0 ? rr.starts[next_start - 1] : 0;  // the last row that begins a new range
            const auto per_row = [&](int e) { return (3 + 2 * tiles(rr.hi[e - 1] - rr.lo[q])) / (double)(e - q); };
            if (cut > q + 1 && per_row(cut) < per_row(end)) end = cut;
        }
        cuts.push_back(end);
    }
    const int n_halves = (int)cuts.size() - 1;
    for (int i = 0; i < n_halves;) {
        bool two = pairs && i + 1 < n_halves;
        if (two && i + 1 >= n_global && i < n_global) {  // a half of the global block with one of table rows
            two = ceil_div(nv, kTile) <= 2 && cuts[i + 1] >= P;
        } else if (two && i >= n_global) {
            const int r0 = cuts[i], r1 = cuts[i + 1], r2 = cuts[i + 2];
            const int both = rr.hi[r2 - 1] - rr.lo[r0];
            const int apart = tiles(rr.hi[r1 - 1] - rr.lo[r0]) + tiles(rr.hi[r2 - 1] - rr.lo[r1]);
            two = 4 * tiles(both) <= 3 * apart || tiles(both) <= 4;
        }
        add(cuts[i], cuts[i + 1], two ? cuts[i + 2] : cuts[i + 1]);
        i += two ? 2 : 1;
    }
}

void list_units(const mate_plan_t *pl, const std::vector<RowRanges> &ranges, bool pairs, bool fill_up, ProtoList &out) {
    out.protos.clear();
    out.tiles.clear();
    size_t rows = 0;
    for (const RowRanges &rr : ranges) rows += rr.nv;
    out.protos.reserve(rows / kTile + 2 * ranges.size());
    out.tiles.reserve(rows / kTile * 8);
    for (int v = 0; v < 2; ++v)
        for (int b = 0; b < pl->B && pl->view[v].n_heads > 0; ++b) add_units(ranges[(size_t)v * pl->B + b], b, v, pairs, fill_up, out);
    sort_protos(out);
}

// Backward: single halves, none split; its work items are the units, once per side.  Longest first: the CTAs of
// the persistent kernel take work from the head of the list as they become free (a shared counter), so the
// order is the whole schedule.
void make_bwd_units(mate_plan_t *pl, const ProtoList &singles, const HeadLists &heads, bool costs) {
    size_t n = 0;
    for (const Proto &pr : singles.protos) n += heads.heads[pr.view].size();
    pl->bwd_units.clear();
    pl->bwd_units.reserve(n);
    for (const Proto &pr : singles.protos)
        for (int h : heads.heads[pr.view]) {
            if (costs) pl->bwd_costs.push_back(pr.cost);
            pl->bwd_units.push_back(pr.u);
            pl->bwd_units.back().hv = mate::pack_hv(h, pr.view);
        }
    pl->n_bwd_units = (int)pl->bwd_units.size();
    pl->bwd_grid = std::min(std::max(pl->n_ctas, 1), std::max(2 * pl->n_bwd_units, pl->n_pads));
}

// Tiles [i0, i1) of a unit (kP = 0) as a unit of its own.
FwdUnit slice_unit(const FwdUnit &u, int i0, int i1) {
    const int nA = u.tiles_a();
    FwdUnit w = u;
    const int a0 = std::min(i0, nA), a1 = std::min(i1, nA), b0 = std::max(i0 - nA, 0), b1 = std::max(i1 - nA, 0);
    w.kA0 = u.kA0 + a0 * kTile;
    w.kA_end = a1 > a0 ? std::min(u.kA_end, u.kA0 + a1 * kTile) : w.kA0;
    w.kB0 = u.kB0 + b0 * u.tB;
    w.kB_end = b1 > b0 ? std::min(u.kB_end, u.kB0 + b1 * u.tB) : w.kB0;
    return w;
}

// Forward.  A unit of more than 1.3 of a CTA's share of the clocks is cut between tiles into parts of about
// 0.75 of it (never less than four tiles), to be combined in the kernel; longest first, as for the backward.
void make_fwd_units(mate_plan_t *pl, const std::vector<RowRanges> &ranges, const HeadLists &heads, bool costs) {
    const int n_ctas = std::max(pl->n_ctas, 1);
    ProtoList list;
    list_units(pl, ranges, true, false, list);
    size_t n_inst = 0;
    for (const Proto &pr : list.protos) n_inst += heads.heads[pr.view].size();
    // Single halves when there are not enough pairs for half of the SMs: a CTA then works on one half only,
    // which takes less than the time of both.
    if (2 * (int)n_inst <= n_ctas) list_units(pl, ranges, false, false, list);
    int64_t total = 0;
    for (const Proto &pr : list.protos) total += pr.cost * (int64_t)heads.heads[pr.view].size();
    const int64_t share = std::max<int64_t>(total / n_ctas, 1);

    struct Entry {
        FwdUnit u;
        int view;
        int64_t cost;
    };
    std::vector<Entry> entries;
    entries.reserve(list.protos.size());
    size_t ws_bytes = 0;
    pl->n_fwd_slots = 0;
    size_t n_units = 0;
    for (const Proto &pr : list.protos) {
        const size_t n_heads = heads.heads[pr.view].size();
        int parts = 1;
        if (pr.u.kP() == 0 && 10 * pr.cost > 13 * share)
            parts = (int)std::max<int64_t>(1, std::min<int64_t>(pr.n_tiles / 4, (4 * pr.cost + 3 * share - 1) / (3 * share)));
        if (parts == 1) {
            entries.push_back({pr.u, pr.view, pr.cost});
        } else {
            const int32_t *tile = list.tiles.data() + pr.tile0;
            for (int part = 0; part < parts; ++part) {
                const int i0 = (int)((int64_t)pr.n_tiles * part / parts), i1 = (int)((int64_t)pr.n_tiles * (part + 1) / parts);
                Entry e{slice_unit(pr.u, i0, i1), pr.view, kUnitClk + kPartClk};
                for (int i = i0; i < i1; ++i) e.cost += tile[i];
                e.u.parts = parts | part << 16;
                e.u.ctr = pl->n_fwd_slots;  // of the first head; the others follow
                e.u.ws_off = (int32_t)((ws_bytes + part * mate::kPartialBytes) >> 10);
                entries.push_back(e);
            }
            pl->n_fwd_slots += (int)n_heads;
            ws_bytes += n_heads * parts * mate::kPartialBytes;
        }
        n_units += n_heads * parts;
    }
    std::stable_sort(entries.begin(), entries.end(), [](const Entry &a, const Entry &b) { return a.cost > b.cost; });
    pl->fwd_units.clear();
    pl->fwd_units.reserve(n_units);
    for (const Entry &e : entries) {
        int k = 0;
        for (int h : heads.heads[e.view]) {
            if (costs) pl->fwd_costs.push_back(e.cost);
            pl->fwd_units.push_back(e.u);
            FwdUnit &u = pl->fwd_units.back();
            u.hv = mate::pack_hv(h, e.view);
            if (u.n_parts() > 1) {
                u.ctr += k;
                u.ws_off += (int32_t)((k * u.n_parts() * mate::kPartialBytes) >> 10);
            }
            ++k;
        }
    }
    pl->n_fwd_units = (int)pl->fwd_units.size();
    pl->fwd_ws_bytes = ws_bytes;
    // padding rows of every (example, head)
    pl->pads.clear();
    for (int b = 0; b < pl->B; ++b)
        for (int t0 = pl->n_valid[b]; t0 < pl->N; t0 += mate::kPadRows)
            for (int h = 0; h < pl->H; ++h) pl->pads.push_back({b, mate::pack_hv(h, pl->head_view[h]), t0, std::min(mate::kPadRows, pl->N - t0)});
    pl->n_pads = (int)pl->pads.size();
    pl->fwd_grid = std::min(n_ctas, std::max(pl->n_fwd_units, pl->n_pads));
    if (getenv("MATE_LOG"))
        fprintf(stderr, "[mate] forward: %d units (%d split), %d CTAs, estimated clocks per CTA %lld, largest unit %lld; workspace %zu "
                        "bytes; %d chunks of padding\n",
                pl->n_fwd_units, pl->n_fwd_slots, pl->fwd_grid, (long long)share,
                entries.empty() ? 0ll : (long long)entries.front().cost, pl->fwd_ws_bytes, pl->n_pads);
}

// costs: the lists are to be joined with others (join_units).
void build_units(mate_plan_t *pl, const int32_t *const (&seg_off_host)[2], bool costs) {
    static_assert(mate::kPartialBytes % 1024 == 0, "ws_off counts KiB");
    std::vector<RowRanges> ranges((size_t)2 * pl->B);
    for (int v = 0; v < 2; ++v)
        for (int b = 0; b < pl->B && pl->view[v].n_heads > 0; ++b) fill_ranges(pl, seg_off_host, v, b, ranges[(size_t)v * pl->B + b]);
    // unmasked pairs per (example, view): the global block with everything, every table row with the block and
    // its own range
    pl->pairs.assign((size_t)pl->B * 2, 0);
    for (int v = 0; v < 2; ++v)
        for (int b = 0; b < pl->B && pl->view[v].n_heads > 0; ++b) {
            const RowRanges &rr = ranges[(size_t)v * pl->B + b];
            pl->pairs[(size_t)b * 2 + v] = (int64_t)rr.P * rr.nv + (int64_t)rr.P * (rr.nv - rr.P) + rr.own;
        }

    const HeadLists heads(pl);
    make_fwd_units(pl, ranges, heads, costs);
    size_t n_halves = 0;
    for (int v = 0; v < 2; ++v)
        for (int b = 0; b < pl->B; ++b) n_halves += heads.heads[v].size() * ceil_div(ranges[(size_t)v * pl->B + b].nv, kTile);
    ProtoList singles;
    list_units(pl, ranges, false, n_halves > (size_t)std::max(pl->n_ctas, 1), singles);
    make_bwd_units(pl, singles, heads, costs);
}

// Row-or-column plan: the lists of the two further passes join this plan's, longest first again, so that one launch
// does all three (they are independent until their results are merged).
void join_units(mate_plan_t *pl) {
    int slots = pl->n_fwd_slots;
    const auto by_cost = [](std::vector<FwdUnit> &units, std::vector<int64_t> &costs) {
        std::vector<int> order(units.size());
        for (size_t i = 0; i < order.size(); ++i) order[i] = (int)i;
        std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return costs[a] > costs[b]; });
        std::vector<FwdUnit> u(units.size());
        std::vector<int64_t> c(units.size());
        for (size_t i = 0; i < order.size(); ++i) {
            u[i] = units[order[i]];
            c[i] = costs[order[i]];
        }
        units.swap(u);
        costs.swap(c);
    };
    for (int s = 0; s < 2; ++s) {
        mate_plan_t *sub = pl->sub[s];
        const auto view = [s](int32_t hv) { return mate::pack_hv(mate::head_of(hv), 2 + s); };
        for (FwdUnit u : sub->fwd_units) {
            u.hv = view(u.hv);
            if (u.n_parts() > 1) {
                u.ctr += slots;
                u.ws_off += (int32_t)(pl->fwd_ws_bytes >> 10);
            }
            pl->fwd_units.push_back(u);
        }
        for (FwdUnit u : sub->bwd_units) {
            u.hv = view(u.hv);
            pl->bwd_units.push_back(u);
        }
        for (mate::PadChunk c : sub->pads) {
            c.hv = view(c.hv);
            pl->pads.push_back(c);
        }
        pl->fwd_costs.insert(pl->fwd_costs.end(), sub->fwd_costs.begin(), sub->fwd_costs.end());
        pl->bwd_costs.insert(pl->bwd_costs.end(), sub->bwd_costs.begin(), sub->bwd_costs.end());
        slots += sub->n_fwd_slots;
        pl->fwd_ws_bytes += sub->fwd_ws_bytes;
    }
    by_cost(pl->fwd_units, pl->fwd_costs);
    by_cost(pl->bwd_units, pl->bwd_costs);
    for (mate_plan_t *x : {pl, pl->sub[0], pl->sub[1]}) x->fwd_costs = x->bwd_costs = {};
    pl->n_fwd_slots = slots;
    pl->n_fwd_units = (int)pl->fwd_units.size();
    pl->n_bwd_units = (int)pl->bwd_units.size();
    pl->n_pads = (int)pl->pads.size();
    const int n_ctas = std::max(pl->n_ctas, 1);
    pl->fwd_grid = std::min(n_ctas, std::max(pl->n_fwd_units, pl->n_pads));
    pl->bwd_grid = std::min(n_ctas, std::max(2 * pl->n_bwd_units, pl->n_pads));
}

// Device copy of the lists, in one piece: units, padding, arrival counters (zeros; the kernel resets them).
int upload_units(mate_plan_t *pl, cudaStream_t st) {
    const auto lay_out = [pl](char *base) {
        Carver c(base);
        pl->fwd_units_dev = c.take<FwdUnit>(pl->n_fwd_units);
        pl->bwd_units_dev = c.take<FwdUnit>(pl->n_bwd_units);
        pl->pads_dev = c.take<mate::PadChunk>(pl->n_pads);
        pl->fwd_counters_dev = c.take<int32_t>(mate::kSchedWords + 8 * (size_t)pl->n_fwd_slots);
        return align_up(c.off, 256);
    };
    const size_t bytes = lay_out(nullptr);
    mate::Staging host;
    if (!mate::staging_take(bytes, pl->device, &host)) return MATE_ERR_NOMEM;
    if (!mate::pool_take(bytes, st, pl->device, &pl->work_block)) {
        mate::staging_give(host, st);
        return MATE_ERR_NOMEM;
    }
    lay_out((char *)host.ptr);
    std::copy(pl->fwd_units.begin(), pl->fwd_units.end(), pl->fwd_units_dev);
    std::copy(pl->bwd_units.begin(), pl->bwd_units.end(), pl->bwd_units_dev);
    std::copy(pl->pads.begin(), pl->pads.end(), pl->pads_dev);
    std::fill_n(pl->fwd_counters_dev, mate::kSchedWords + 8 * (size_t)pl->n_fwd_slots, 0);
    lay_out((char *)pl->work_block.ptr);
    bool ok = cudaMemcpyAsync(pl->work_block.ptr, host.ptr, bytes, cudaMemcpyHostToDevice, st) == cudaSuccess;
    mate::staging_give(host, st);
    ok = ok && cudaEventCreateWithFlags(&pl->ready, cudaEventDisableTiming) == cudaSuccess &&
         cudaEventRecord(pl->ready, st) == cudaSuccess;
    if (!ok) return MATE_ERR_CUDA;
    return MATE_OK;
}

}  // namespace

extern "C" {

const char *mate_status_string(int status) {
    switch (status) {
        case MATE_OK: return "ok";
        case MATE_ERR_INVALID_ARG: return "invalid argument";
        case MATE_ERR_UNSUPPORTED: return "unsupported head dim, dtype or implementation";
        case MATE_ERR_ALIGNMENT: return "tensor pointer not 16-byte aligned";
        case MATE_ERR_CUDA: return "CUDA runtime error";
        case MATE_ERR_TIMEOUT: return "bounded device wait expired";
        case MATE_ERR_NOMEM: return "out of memory";
        case MATE_ERR_WORKSPACE: return "workspace missing or too small";
        case MATE_ERR_TOO_LARGE: return "B*H*N exceeds the built-in scratch of mate_attn_bwd_noalloc";
        default: return "unknown status";
    }
}

int mate_plan_destroy(mate_plan_t *plan) {
    if (!plan) return MATE_OK;
    for (int s = 0; s < 2; ++s) mate_plan_destroy(plan->sub[s]);
    const uint64_t stream = plan->elsewhere ? 0 : plan->stream;
    mate::pool_give(plan->extra_block, stream);
    mate::pool_give(plan->dev_block, stream);
    mate::pool_give(plan->work_block, stream);
    if (plan->ready) cudaEventDestroy(plan->ready);
    delete plan;
    return MATE_OK;
}

int mate_plan(const int32_t *row_ids, const int32_t *col_ids, int B, int N, int prefix_len,
              const uint8_t *head_view, int H, int max_row_id, int max_col_id, void *stream,
              mate_plan_t **out) {
    return mate_plan_bucketed(row_ids, col_ids, B, N, prefix_len, head_view, H, max_row_id, max_col_id, 0,
                              stream, out);
}

int mate_plan_bucketed(const int32_t *row_ids, const int32_t *col_ids, int B, int N, int prefix_len,
                       const uint8_t *head_view, int H, int max_row_id, int max_col_id, int radius,
                       void *stream, mate_plan_t **out) {
    if (out) *out = nullptr;
    if (B <= 0) return MATE_ERR_INVALID_ARG;
    return no_throw([&]() {
        const std::vector<int32_t> prefix((size_t)B, prefix_len);
        return mate_plan_varlen(row_ids, col_ids, B, N, prefix.data(), head_view, H, max_row_id, max_col_id, radius,
                                stream, out);
    });
}

static int build_plan(const int32_t *row_ids, const int32_t *col_ids, int B, int N, const int32_t *prefix_len,
                      const int32_t *global_len, const uint8_t *head_view, int H, int max_row_id, int max_col_id,
                      int radius, int bounds_mode, int group, bool upload, void *stream, mate_plan_t **out);

int mate_plan_varlen(const int32_t *row_ids, const int32_t *col_ids, int B, int N, const int32_t *prefix_len,
                     const uint8_t *head_view, int H, int max_row_id, int max_col_id, int radius,
                     void *stream, mate_plan_t **out) {
    return build_plan(row_ids, col_ids, B, N, prefix_len, nullptr, head_view, H, max_row_id, max_col_id, radius,
                      mate::kBoundsOwn, 1, true, stream, out);
}

int mate_plan_bucketed_global(const int32_t *row_ids, const int32_t *col_ids, int B, int N, const int32_t *prefix_len,
                              const int32_t *global_len, const uint8_t *head_view, int H, int max_row_id,
                              int max_col_id, int radius, void *stream, mate_plan_t **out) {
    if (out) *out = nullptr;
    if (!global_len || !prefix_len || B <= 0 || radius <= 0) return MATE_ERR_INVALID_ARG;
    for (int b = 0; b < B; ++b)
        if (global_len[b] < prefix_len[b] || global_len[b] > N) return MATE_ERR_INVALID_ARG;
    return build_plan(row_ids, col_ids, B, N, prefix_len, global_len, head_view, H, max_row_id, max_col_id, radius,
                      mate::kBoundsOwn, 1, true, stream, out);
}

/* Packed batches: the examples lie one behind the other on a common token axis.  The plan itself is the
 * padded one over N = the longest example (small integer arrays); what changes is where the kernels
 * find an example's rows in the tensors, and that positions behind an example's end do not exist. */
static int plan_packed(const int32_t *row_ids, const int32_t *col_ids, int B, const int32_t *cu_seqlens,
                       const int32_t *prefix_len, const uint8_t *head_view, int H, int max_row_id, int max_col_id,
                       void *stream, mate_plan_t **out) {
    if (!row_ids || !col_ids || !cu_seqlens || !prefix_len || !head_view || !out || B <= 0 || H <= 0)
        return MATE_ERR_INVALID_ARG;
    if (cu_seqlens[0] != 0) return MATE_ERR_INVALID_ARG;
    int n_max = 1;
    std::vector<int32_t> off_len((size_t)2 * B);
    for (int b = 0; b < B; ++b) {
        const int len = cu_seqlens[b + 1] - cu_seqlens[b];
        if (len < 0 || prefix_len[b] < 0 || prefix_len[b] > len) return MATE_ERR_INVALID_ARG;
        n_max = std::max(n_max, len);
        off_len[b] = cu_seqlens[b];
        off_len[B + b] = len;
    }
    const int T = cu_seqlens[B];
    cudaStream_t st = (cudaStream_t)stream;
    const size_t BN = (size_t)B * n_max;
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess) return MATE_ERR_CUDA;
    mate::Block offs, ids;
    mate::Staging host;
    bool ok = mate::staging_take(sizeof(int32_t) * 2 * B, dev, &host) && mate::pool_take(sizeof(int32_t) * 2 * B, st, dev, &offs) &&
              mate::pool_take(sizeof(int32_t) * 2 * BN, st, dev, &ids);
    int rc = ok ? MATE_OK : MATE_ERR_NOMEM;
    mate_plan_t *pl = nullptr;
    const uint64_t id = mate::stream_id(st);
    int32_t *off_dev = (int32_t *)offs.ptr, *ids_dev = (int32_t *)ids.ptr;
    if (ok) {
        std::copy(off_len.begin(), off_len.end(), (int32_t *)host.ptr);
        ok = cudaMemcpyAsync(off_dev, host.ptr, sizeof(int32_t) * 2 * B, cudaMemcpyHostToDevice, st) == cudaSuccess &&
             mate::launch_unpack_ids(row_ids, col_ids, B, n_max, off_dev, off_dev + B, ids_dev, ids_dev + BN, st) == cudaSuccess;
        rc = ok ? build_plan(ids_dev, ids_dev + BN, B, n_max, prefix_len, nullptr, head_view, H, max_row_id, max_col_id, 0,
                             mate::kBoundsOwn, 1, true, stream, &pl)
                : MATE_ERR_CUDA;
    }
    mate::staging_give(host, st);
    mate::pool_give(ids, id);
    if (rc != MATE_OK) {
        mate::pool_give(offs, id);
        return rc;
    }
    pl->extra_block = offs;
    pl->T = T;
    pl->tok_off_dev = off_dev;
    pl->len_dev = off_dev + B;
    *out = pl;
    return MATE_OK;
}

int mate_plan_packed(const int32_t *row_ids, const int32_t *col_ids, int B, const int32_t *cu_seqlens,
                     const int32_t *prefix_len, const uint8_t *head_view, int H, int max_row_id, int max_col_id,
                     void *stream, mate_plan_t **out) {
    if (out) *out = nullptr;
    return no_throw([&]() {
        return plan_packed(row_ids, col_ids, B, cu_seqlens, prefix_len, head_view, H, max_row_id, max_col_id, stream, out);
    });
}

/* The head-independent pattern: three passes over plans the ordinary kernels can run (see mate.h).
 *   main plan  every head a row head: prefix rows against everything, table rows against the prefix
 *              and their own row (which holds their own cell)
 *   sub[0]     ids = (column, row) pairs, column-major, prefix treated as padding: table rows against
 *              the cells of their column in front of their own cell
 *   sub[1]     the same behind their own cell
 * The three key sets of a row are disjoint and their union is the pattern. */
static int plan_sat(const int32_t *row_ids, const int32_t *col_ids, int B, int N, int prefix_len, int H,
                    int max_row_id, int max_col_id, void *stream, mate_plan_t **out) {
    if (!out || B <= 0 || H <= 0 || max_row_id < 0 || max_col_id < 0) return MATE_ERR_INVALID_ARG;
    if ((long long)(max_row_id + 1) * (max_col_id + 1) > (1ll << 28)) return MATE_ERR_UNSUPPORTED;
    const std::vector<int32_t> prefix((size_t)B, prefix_len), zero((size_t)B, 0);
    const std::vector<uint8_t> rows_only((size_t)H, 0), cols_only((size_t)H, 1);
    mate_plan_t *pl = nullptr;
    int rc = build_plan(row_ids, col_ids, B, N, prefix.data(), nullptr, rows_only.data(), H, max_row_id, max_col_id, 0,
                        mate::kBoundsOwn, 1, false, stream, &pl);
    if (rc != MATE_OK) return rc;
    cudaStream_t st = (cudaStream_t)stream;
    const int n_row_ids = max_row_id + 1, max_pair = n_row_ids * (max_col_id + 1) - 1;
    bool ok = mate::pool_take(sizeof(int32_t) * (size_t)B * N, st, pl->device, &pl->extra_block);
    pl->pair_ids_dev = (int32_t *)pl->extra_block.ptr;
    ok = ok && mate::launch_pair_ids(row_ids, col_ids, B, N, pl->prefix_dev, n_row_ids, pl->pair_ids_dev, st) == cudaSuccess;
    if (!ok) {
        cudaGetLastError();
        mate_plan_destroy(pl);
        return MATE_ERR_NOMEM;
    }
    for (int s = 0; s < 2 && rc == MATE_OK; ++s)
        rc = build_plan(pl->pair_ids_dev, pl->pair_ids_dev, B, N, zero.data(), nullptr, cols_only.data(), H, max_pair, max_pair, 0,
                        s == 0 ? mate::kBoundsBefore : mate::kBoundsAfter, n_row_ids, false, stream, &pl->sub[s]);
    if (rc == MATE_OK)
        rc = no_throw([&]() {
            join_units(pl);
            return upload_units(pl, st);
        });
    if (rc != MATE_OK) {
        mate_plan_destroy(pl);
        return rc;
    }
    *out = pl;
    return MATE_OK;
}

int mate_plan_sat(const int32_t *row_ids, const int32_t *col_ids, int B, int N, int prefix_len, int H,
                  int max_row_id, int max_col_id, void *stream, mate_plan_t **out) {
    if (out) *out = nullptr;
    return no_throw([&]() { return plan_sat(row_ids, col_ids, B, N, prefix_len, H, max_row_id, max_col_id, stream, out); });
}

// Fills an empty plan from checked arguments; the caller owns the plan and the staging buffer whatever comes of it.
static int fill_plan(mate_plan_t *pl, mate::Staging &host, const int32_t *row_ids, const int32_t *col_ids, int B, int N,
                     const int32_t *prefix_len, const int32_t *global_len, const uint8_t *head_view, int H, int max_row_id,
                     int max_col_id, int radius, int bounds_mode, int group, bool upload, cudaStream_t st) {
    pl->B = B;
    pl->N = N;
    pl->prefix.assign(prefix_len, prefix_len + B);
    if (global_len) pl->global.assign(global_len, global_len + B);
    else pl->global = pl->prefix;
    pl->H = H;
    pl->radius = radius;
    pl->bounds_mode = bounds_mode;
    pl->group = std::max(group, 1);
    pl->head_view.assign(head_view, head_view + H);
    pl->view[0].max_id = max_row_id;
    pl->view[1].max_id = max_col_id;
    for (int h = 0; h < H; ++h) pl->view[head_view[h]].n_heads++;

    {
        int dev = 0;
        if (cudaGetDevice(&dev) != cudaSuccess ||
            cudaDeviceGetAttribute(&pl->n_ctas, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
            return MATE_ERR_CUDA;
        pl->device = dev;
    }
    pl->stream = mate::stream_id(st);
    if (pl->stream == 0) pl->elsewhere = true;
    const PlanLayout L = carve(pl, nullptr);
    if (!mate::staging_take(std::max(L.in_bytes, L.out_bytes), pl->device, &host) ||
        !mate::pool_take(L.total, st, pl->device, &pl->dev_block))
        return MATE_ERR_NOMEM;
    char *dev_base = (char *)pl->dev_block.ptr, *host_base = (char *)host.ptr;
    carve(pl, dev_base);
    const auto in_host = [&](const void *dev) { return host_base + ((const char *)dev - dev_base - L.in_off); };
    memset(host_base, 0, L.in_bytes);
    memcpy(in_host(pl->prefix_dev), pl->prefix.data(), B * sizeof(int32_t));
    memcpy(in_host(pl->global_dev), pl->global.data(), B * sizeof(int32_t));
    memcpy(in_host(pl->head_view_dev), pl->head_view.data(), H);
    bool ok = cudaMemcpyAsync(dev_base + L.in_off, host_base, L.in_bytes, cudaMemcpyHostToDevice, st) == cudaSuccess;
    ok = ok && mate::launch_plan_kernels(row_ids, col_ids, B, N, pl->prefix_dev, pl->global_dev, radius, bounds_mode, pl->group,
                                         pl->view[0], pl->view[1], pl->n_valid_dev, pl->status_dev, st) == cudaSuccess;
    ok = ok && cudaMemcpyAsync(host_base, dev_base + L.out_off, L.out_bytes, cudaMemcpyDeviceToHost, st) == cudaSuccess;
    ok = ok && cudaStreamSynchronize(st) == cudaSuccess;
    if (!ok) return MATE_ERR_CUDA;
    const auto out_host = [&](const void *dev) { return (const int32_t *)(host_base + ((const char *)dev - dev_base - L.out_off)); };
    if (out_host(pl->status_dev)[0] != 0) return MATE_ERR_INVALID_ARG;
    pl->n_valid.assign(out_host(pl->n_valid_dev), out_host(pl->n_valid_dev) + B);
    const int32_t *seg_off_host[2] = {out_host(pl->view[0].seg_off), out_host(pl->view[1].seg_off)};
    build_units(pl, seg_off_host, !upload);
    return upload ? upload_units(pl, st) : MATE_OK;
}

static int build_plan(const int32_t *row_ids, const int32_t *col_ids, int B, int N, const int32_t *prefix_len,
                      const int32_t *global_len, const uint8_t *head_view, int H, int max_row_id, int max_col_id,
                      int radius, int bounds_mode, int group, bool upload, void *stream, mate_plan_t **out) {
    if (out) *out = nullptr;
    if (radius < 0) return MATE_ERR_INVALID_ARG;
    if (!row_ids || !col_ids || !head_view || !out || !prefix_len) return MATE_ERR_INVALID_ARG;
    if (B <= 0 || N <= 0 || H <= 0) return MATE_ERR_INVALID_ARG;
    for (int b = 0; b < B; ++b)
        if (prefix_len[b] < 0 || prefix_len[b] > N) return MATE_ERR_INVALID_ARG;
    if (max_row_id < 0 || max_col_id < 0) return MATE_ERR_INVALID_ARG;
    if ((long long)B * N > (1ll << 30) || max_row_id > (1 << 28) || max_col_id > (1 << 28) || H >= 1 << mate::kViewShift)
        return MATE_ERR_UNSUPPORTED;
    for (int h = 0; h < H; ++h)
        if (head_view[h] > 1) return MATE_ERR_INVALID_ARG;

    cudaStream_t st = (cudaStream_t)stream;
    mate_plan_t *pl = new (std::nothrow) mate_plan_t();
    if (!pl) return MATE_ERR_NOMEM;
    mate::Staging host;
    const int rc = no_throw([&]() {
        return fill_plan(pl, host, row_ids, col_ids, B, N, prefix_len, global_len, head_view, H, max_row_id, max_col_id, radius,
                         bounds_mode, group, upload, st);
    });
    mate::staging_give(host, st);
    if (rc != MATE_OK) {
        mate_plan_destroy(pl);
        return rc;
    }
    *out = pl;
    return MATE_OK;
}

int mate_plan_get(const mate_plan_t *plan, int view, int32_t *perm, int32_t *inv_perm,
                  int32_t *seg_off) {
    if (!plan || view < 0 || view > 1) return MATE_ERR_INVALID_ARG;
    const ViewPlan &vp = plan->view[view];
    const size_t BN = (size_t)plan->B * plan->N * sizeof(int32_t);
    bool ok = true;
    if (perm) ok = ok && cudaMemcpy(perm, vp.perm, BN, cudaMemcpyDeviceToHost) == cudaSuccess;
    if (inv_perm) ok = ok && cudaMemcpy(inv_perm, vp.inv_perm, BN, cudaMemcpyDeviceToHost) == cudaSuccess;
    if (seg_off)
        ok = ok && cudaMemcpy(seg_off, vp.seg_off, (size_t)plan->B * (vp.max_id + 2) * sizeof(int32_t),
                              cudaMemcpyDeviceToHost) == cudaSuccess;
    return ok ? MATE_OK : MATE_ERR_CUDA;
}

int mate_plan_useful_pairs(const mate_plan_t *plan, int64_t *pairs) {
    if (!plan || !pairs) return MATE_ERR_INVALID_ARG;
    for (int b = 0; b < plan->B; ++b)
        for (int h = 0; h < plan->H; ++h) {
            int64_t c = plan->pairs[(size_t)b * 2 + plan->head_view[h]];
            for (int s = 0; s < 2; ++s)
                if (plan->sub[s]) c += plan->sub[s]->pairs[(size_t)b * 2 + 1];
            pairs[(size_t)b * plan->H + h] = c;
        }
    return MATE_OK;
}

int mate_plan_status(const mate_plan_t *plan, void *stream) {
    if (!plan) return MATE_ERR_INVALID_ARG;
    for (int s = 0; s < 2; ++s)
        if (plan->sub[s]) {
            const int rc = mate_plan_status(plan->sub[s], stream);
            if (rc != MATE_OK) return rc;
        }
    cudaStream_t st = (cudaStream_t)stream;
    if (mate::use_plan(plan, st) != cudaSuccess) return MATE_ERR_CUDA;
    int32_t s[4] = {0, 0, 0, 0};
    if (cudaMemcpyAsync(s, plan->status_dev, sizeof(s), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
        cudaMemsetAsync(plan->status_dev + 1, 0, 2 * sizeof(int32_t), st) != cudaSuccess ||
        cudaStreamSynchronize(st) != cudaSuccess)
        return MATE_ERR_CUDA;
    if (s[1] != 0) {
        if (getenv("MATE_LOG")) fprintf(stderr, "[mate] a bounded wait expired\n");
        // a kernel that gave up may have left the arrival counters half way
        // (the passes of a row-or-column plan have none of their own)
        if (plan->fwd_counters_dev &&
            (cudaMemsetAsync(plan->fwd_counters_dev, 0, sizeof(int32_t) * (mate::kSchedWords + 8 * (size_t)plan->n_fwd_slots), st) != cudaSuccess ||
             cudaStreamSynchronize(st) != cudaSuccess))
            return MATE_ERR_CUDA;
        return MATE_ERR_TIMEOUT;
    }
    return MATE_OK;
}

// The plan's arrays, its CTA count and the kernels' per-device set-up belong to the device the plan
// was made on: a call with another device current is refused before anything is launched.
static int check_device(const mate_plan_t *plan) {
    int dev = -1;
    if (cudaGetDevice(&dev) != cudaSuccess) return MATE_ERR_CUDA;
    return dev == plan->device ? MATE_OK : MATE_ERR_INVALID_ARG;
}

static int check_common(const mate_plan_t *plan, int d, int dtype, unsigned flags, bool *use_tc) {
    if (!plan) return MATE_ERR_INVALID_ARG;
    if (dtype != MATE_BF16 && dtype != MATE_F32) return MATE_ERR_UNSUPPORTED;
    if (d <= 0 || d % 8 != 0 || d > 128) return MATE_ERR_UNSUPPORTED;
    const unsigned impl = flags & 3u;
    constexpr unsigned kLoaderBits = MATE_FLAG_BULK_TILES | MATE_FLAG_GATHER_TILES;
    if (impl == 3u || (flags & ~(3u | MATE_FLAG_VIEW_ORDER | kLoaderBits)) || (flags & kLoaderBits) == kLoaderBits)
        return MATE_ERR_INVALID_ARG;
    const bool tc_ok = mate::tc_supported(d, dtype);
    if (impl == MATE_IMPL_TCGEN05 && !tc_ok) return MATE_ERR_UNSUPPORTED;
    *use_tc = (impl == MATE_IMPL_TCGEN05) || (impl == MATE_IMPL_AUTO && tc_ok);
    return MATE_OK;
}

// Scratch of the ordinary kernels and of a whole call.  For a row-or-column plan the call holds, behind the kernels'
// own scratch (the tensor-core kernels do the three passes in one launch; without tensor cores they run one after
// the other and share it), the outputs of the two extra passes: forward 2 x (O + LSE), backward 2 x (dQ, dK, dV).
static size_t pass_fwd_bytes(const mate_plan_t *plan, int d, bool use_tc) {
    return align_up(use_tc ? mate::tc_fwd_workspace(plan, d) : 0, 256);
}
static size_t pass_bwd_bytes(const mate_plan_t *plan, bool use_tc) {
    return align_up(use_tc ? mate::tc_bwd_workspace(plan) : mate::simt_bwd_workspace(plan), 256);
}
static size_t elem_bytes(int dtype) { return dtype == MATE_F32 ? 4 : 2; }

int mate_attn_workspace_bytes(const mate_plan_t *plan, int d, int dtype, unsigned flags,
                              size_t *fwd_bytes, size_t *bwd_bytes) {
    bool use_tc = false;
    int rc = check_common(plan, d, dtype, flags, &use_tc);
    if (rc != MATE_OK) return rc;
    const size_t rows = plan->n_rows();
    size_t f = pass_fwd_bytes(plan, d, use_tc), b = pass_bwd_bytes(plan, use_tc);
    if (plan->sub[0]) {
        f += 2 * (align_up(rows * d * elem_bytes(dtype), 256) + align_up(rows * sizeof(float), 256));
        b += 6 * align_up(rows * d * elem_bytes(dtype), 256);
    }
    if (fwd_bytes) *fwd_bytes = f;
    if (bwd_bytes) *bwd_bytes = b;
    return MATE_OK;
}

static cudaError_t use_plans(const mate_plan_t *plan, cudaStream_t st) {
    cudaError_t rc = mate::use_plan(plan, st);
    for (int s = 0; s < 2 && rc == cudaSuccess; ++s)
        if (plan->sub[s]) rc = mate::use_plan(plan->sub[s], st);
    return rc;
}

int mate_attn_fwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V, int d,
                  int dtype, float scale, void *O, float *LSE, void *workspace,
                  size_t workspace_bytes, unsigned flags, void *stream) {
    bool use_tc = false;
    int rc = check_common(plan, d, dtype, flags, &use_tc);
    if (rc != MATE_OK) return rc;
    if ((rc = check_device(plan)) != MATE_OK) return rc;
    if (!Q || !K || !V || !O || !LSE) return MATE_ERR_INVALID_ARG;
    if (!aligned16(Q) || !aligned16(K) || !aligned16(V) || !aligned16(O) || !aligned16(LSE))
        return MATE_ERR_ALIGNMENT;
    cudaStream_t st = (cudaStream_t)stream;
    // the tensor-core forward takes the row maximum before scaling, which needs scale > 0
    if (use_tc && !(scale > 0.f)) {
        if ((flags & 3u) == MATE_IMPL_TCGEN05) return MATE_ERR_UNSUPPORTED;
        use_tc = false;
    }
    size_t need = 0;
    mate_attn_workspace_bytes(plan, d, dtype, use_tc ? MATE_IMPL_TCGEN05 : MATE_IMPL_SIMT, &need, nullptr);
    if (need > 0 && (!workspace || workspace_bytes < need)) return MATE_ERR_WORKSPACE;
    if (need > 0 && (reinterpret_cast<uintptr_t>(workspace) & 255u)) return MATE_ERR_ALIGNMENT;
    if ((flags & MATE_FLAG_VIEW_ORDER) && (plan->sub[0] || plan->T)) return MATE_ERR_UNSUPPORTED;
    if (use_plans(plan, st) != cudaSuccess) return MATE_ERR_CUDA;
    // Row-or-column pattern: the two passes over the rest of the column, and then the merge.
    const size_t rows = plan->n_rows();
    const size_t o_bytes = align_up(rows * d * elem_bytes(dtype), 256), l_bytes = align_up(rows * sizeof(float), 256);
    char *w = (char *)workspace + pass_fwd_bytes(plan, d, use_tc);
    void *Os[mate::kPasses] = {O, nullptr, nullptr};
    float *Ls[mate::kPasses] = {LSE, nullptr, nullptr};
    for (int i = 1; i < mate::kPasses && plan->sub[0]; ++i, w += o_bytes + l_bytes) {
        Os[i] = w;
        Ls[i] = (float *)(w + o_bytes);
    }
    if (use_tc) {  // all passes at once
        rc = mate::tc_fwd(plan, Q, K, V, scale, Os, Ls, workspace, flags, st);
    } else {
        for (int i = 0; i < mate::kPasses && rc == MATE_OK; ++i)
            if (const mate_plan_t *pass = i ? plan->sub[i - 1] : plan)
                rc = mate::simt_fwd(pass, Q, K, V, d, dtype, scale, Os[i], Ls[i], flags, st);
    }
    if (rc != MATE_OK || !plan->sub[0]) return rc;
    return mate::launch_merge_passes(O, LSE, Os[1], Ls[1], Os[2], Ls[2], rows, d, dtype, st) == cudaSuccess ? MATE_OK
                                                                                                           : MATE_ERR_CUDA;
}

int mate_attn_bwd(const mate_plan_t *plan, const void *Q, const void *K, const void *V,
                  const void *O, const float *LSE, const void *dO, int d, int dtype, float scale,
                  void *dQ, void *dK, void *dV, void *workspace, size_t workspace_bytes,
                  unsigned flags, void *stream) {
    bool use_tc = false;
    int rc = check_common(plan, d, dtype, flags, &use_tc);
    if (rc != MATE_OK) return rc;
    if ((rc = check_device(plan)) != MATE_OK) return rc;
    if (!Q || !K || !V || !O || !LSE || !dO || !dQ || !dK || !dV) return MATE_ERR_INVALID_ARG;
    if (flags & MATE_FLAG_VIEW_ORDER) return MATE_ERR_UNSUPPORTED;  // forward only
    const void *ptrs[] = {Q, K, V, O, LSE, dO, dQ, dK, dV};
    for (const void *p : ptrs)
        if (!aligned16(p)) return MATE_ERR_ALIGNMENT;
    size_t need = 0;
    mate_attn_workspace_bytes(plan, d, dtype, use_tc ? MATE_IMPL_TCGEN05 : MATE_IMPL_SIMT, nullptr, &need);
    if (!workspace || workspace_bytes < need) return MATE_ERR_WORKSPACE;
    if (reinterpret_cast<uintptr_t>(workspace) & 255u) return MATE_ERR_ALIGNMENT;
    cudaStream_t st = (cudaStream_t)stream;
    if (use_plans(plan, st) != cudaSuccess) return MATE_ERR_CUDA;
    // Row-or-column pattern.  With the final O and LSE every pass computes the gradient of its own
    // pairs.  The two column passes are each other's transpose (keys in front of / behind the own
    // cell), and the kernels take a plan's key ranges for the query side and for the key side alike;
    // run on both plans and summed, every pair is still counted once on each side.
    const size_t n = plan->n_rows() * d;
    const size_t g_bytes = align_up(n * elem_bytes(dtype), 256);
    char *w = (char *)workspace + pass_bwd_bytes(plan, use_tc);
    void *g[3][mate::kPasses] = {{dQ}, {dK}, {dV}};  // of every pass
    for (int i = 1; i < mate::kPasses && plan->sub[0]; ++i)
        for (int t = 0; t < 3; ++t, w += g_bytes) g[t][i] = w;
    if (use_tc) {  // all passes at once
        rc = mate::tc_bwd(plan, Q, K, V, O, LSE, dO, scale, g[0], g[1], g[2], workspace, st);
    } else {
        for (int i = 0; i < mate::kPasses && rc == MATE_OK; ++i)
            if (const mate_plan_t *pass = i ? plan->sub[i - 1] : plan)
                rc = mate::simt_bwd(pass, Q, K, V, O, LSE, dO, d, dtype, scale, g[0][i], g[1][i], g[2][i], workspace, i, st);
    }
    if (rc != MATE_OK || !plan->sub[0]) return rc;
    void *second[3] = {g[0][1], g[1][1], g[2][1]}, *third[3] = {g[0][2], g[1][2], g[2][2]};
    void *outs[3] = {dQ, dK, dV};
    return mate::launch_add3(outs, second, third, n, dtype, st) == cudaSuccess ? MATE_OK : MATE_ERR_CUDA;
}

}  // extern "C"
