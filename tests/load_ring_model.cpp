// The roles of a CTA of the tensor-core kernels as lists of waits and arrivals, run in random interleavings on barriers that
// are waited for by parity, with the barrier slots and parities of csrc/load_ring.h.  Copies and MMA commits arrive on their
// own, any time after they were issued.  Counted: runs in which a wait passes before the phase it is for is over, and runs that
// stand still.
#include <algorithm>
#include <cstdint>
#include <random>
#include <vector>

#include "load_ring.h"

namespace {

constexpr uint32_t kTileBufs = 4, kRecords = 4, kLoadWarps = 4;
using Rows = mate::LoadRing<2>;
using Tiles = mate::LoadRing<kTileBufs>;

struct Barrier {
    int count = 1, pending = 1;
    uint32_t done = 0;  // phases that are over
    void arrive() {
        if (--pending == 0) {
            ++done;
            pending = count;
        }
    }
    bool passes(uint32_t parity) const { return (done & 1) != parity; }
};
struct Op {
    enum Kind { kWait, kArrive, kLater } kind;  // kLater: an arrival that comes by itself
    int bar;
    uint32_t parity = 0;
    int64_t needs = 0;  // phases that have to be over when the wait passes
};
Op wait(int bar, int64_t phase) { return {Op::kWait, bar, (uint32_t)phase & 1, phase + 1}; }  // (phase -1: passes at once)
struct Model {
    std::vector<Barrier> bars;
    std::vector<std::vector<Op>> roles;
    int add(int count) {
        bars.push_back({count, count, 0});
        return (int)bars.size() - 1;
    }
    std::vector<int> add(int n, int count) {
        std::vector<int> v;
        for (int i = 0; i < n; ++i) v.push_back(add(count));
        return v;
    }
    // 1: a wait passed early, 2: the roles stand still, 0: neither
    int run(std::mt19937 &rng) {
        std::vector<size_t> at(roles.size(), 0);
        std::vector<int> later, weight;
        for (size_t i = 0; i < roles.size(); ++i) weight.push_back(rng() % 3 ? 64 : 1 + rng() % 16);  // some roles are slow
        const int later_weight = 1 + rng() % 64;
        for (;;) {
            std::vector<int> ready;
            bool open = !later.empty();
            for (size_t i = 0; i < roles.size(); ++i) {
                if (at[i] >= roles[i].size()) continue;
                open = true;
                const Op &op = roles[i][at[i]];
                if (op.kind != Op::kWait || bars[op.bar].passes(op.parity)) ready.insert(ready.end(), weight[i], (int)i);
            }
            if (!open) return 0;
            if (!later.empty()) ready.insert(ready.end(), later_weight, -1);
            if (ready.empty()) return 2;
            const int who = ready[rng() % ready.size()];
            if (who < 0) {
                const size_t k = rng() % later.size();
                bars[later[k]].arrive();
                later[k] = later.back();
                later.pop_back();
                continue;
            }
            const Op &op = roles[who][at[who]++];
            if (op.kind == Op::kWait) {
                if ((int64_t)bars[op.bar].done < op.needs) return 1;
            } else if (op.kind == Op::kArrive) {
                bars[op.bar].arrive();
            } else {
                later.push_back(op.bar);
            }
        }
    }
};

// Loaders: the rows of every item, then its tiles, in turn by kTeams teams of warps; warp 0 also publishes the records, in the
// forward (`claims`) not before the fourth tile from the end of the item before has been read.
template <uint32_t kTeams>
void loaders(Model &m, const std::vector<int> &tiles, const std::vector<int> &sched_full, const std::vector<int> &sched_empty,
             const std::vector<int> &row_full, const std::vector<int> &row_empty, const std::vector<int> &tile_full,
             const std::vector<int> &tile_empty, bool claims) {
    for (uint32_t w = 0; w < kLoadWarps; ++w) {
        std::vector<Op> ops;
        uint32_t step = 0, c = 0;
        for (uint32_t n = 0; n <= tiles.size(); ++n) {
            if (w == 0) {
                ops.push_back(wait(sched_empty[n % kRecords], (int64_t)(n / kRecords) - 1));
                ops.push_back({Op::kArrive, sched_full[n % kRecords]});
            }
            ops.push_back(wait(sched_full[n % kRecords], n / kRecords));
            ops.push_back({Op::kArrive, sched_empty[n % kRecords]});
            if (n == tiles.size()) break;
            for (int i = -1; i < tiles[n]; ++i, ++step) {
                if (step % kTeams == w * kTeams / kLoadWarps) {
                    const uint32_t load = i < 0 ? n : c;
                    ops.push_back({Op::kWait, i < 0 ? row_empty[Rows::buffer(load)] : tile_empty[Tiles::buffer(load)],
                                   i < 0 ? Rows::wait_parity(load) : Tiles::wait_parity(load), load / (i < 0 ? 2 : kTileBufs)});
                    ops.push_back({Op::kLater, i < 0 ? row_full[Rows::buffer(load)] : tile_full[Tiles::buffer(load)]});
                }
                if (i >= 0) ++c;
            }
            if (claims && w == 0 && tiles[n] > 1) {
                const uint32_t read = c - std::min(tiles[n], 4);
                ops.push_back({Op::kWait, tile_empty[Tiles::buffer(read)], Tiles::wait_parity(read + kTileBufs), read / kTileBufs + 1});
            }
        }
        m.roles.push_back(ops);
    }
}

template <uint32_t kTeams>
Model backward(const std::vector<int> &tiles) {
    Model m;
    const int n_math = 2, n_store = 2, readers = n_math + n_store + 2 + kLoadWarps, parts = kLoadWarps / kTeams;
    const auto sched_full = m.add(kRecords, 1), sched_empty = m.add(kRecords, readers), row_full = m.add(2, parts),
               row_empty = m.add(2, 1 + n_math + n_store), tile_full = m.add(kTileBufs, parts),
               tile_empty = m.add(kTileBufs, 1);
    const int s_full = m.add(1), a_full = m.add(n_math), g_done = m.add(1), st_free = m.add(n_math), item_done = m.add(1), acc_free = m.add(n_store);
    loaders<kTeams>(m, tiles, sched_full, sched_empty, row_full, row_empty, tile_full, tile_empty, false);
    const uint32_t N = (uint32_t)tiles.size();
    const auto record = [&](std::vector<Op> &o, uint32_t n) { o.push_back(wait(sched_full[n % kRecords], n / kRecords)); };
    const auto rows = [&](std::vector<Op> &o, uint32_t n) { o.push_back({Op::kWait, row_full[Rows::buffer(n)], Rows::full_parity(n), n / 2 + 1}); };
    std::vector<Op> math, store, s, g;
    uint32_t c = 0, with_tiles = 0;
    for (uint32_t n = 0; n <= N; ++n) {
        for (auto *o : {&math, &store, &s, &g}) record(*o, n);
        for (auto *o : {&store, &s, &g}) o->push_back({Op::kArrive, sched_empty[n % kRecords]});
        if (n == N) break;
        for (auto *o : {&math, &store, &s}) rows(*o, n);
        store.push_back({Op::kArrive, row_empty[Rows::buffer(n)]});
        if (tiles[n] > 0) {
            g.push_back(wait(acc_free, (int64_t)with_tiles - 1));
            store.push_back(wait(item_done, with_tiles));
            store.push_back({Op::kArrive, acc_free});
            ++with_tiles;
        }
        for (int i = 0; i < tiles[n]; ++i, ++c) {
            s.push_back({Op::kWait, tile_full[Tiles::buffer(c)], Tiles::full_parity(c), c / kTileBufs + 1});
            s.push_back(wait(st_free, (int64_t)c - 1));
            s.push_back({Op::kLater, s_full});
            math.push_back(wait(s_full, c));
            math.push_back({Op::kArrive, st_free});
            math.push_back(wait(g_done, (int64_t)c - 1));
            math.push_back({Op::kArrive, a_full});
            g.push_back(wait(a_full, c));
            g.push_back({Op::kLater, g_done});
            g.push_back({Op::kLater, tile_empty[Tiles::buffer(c)]});
            if (i + 1 == tiles[n]) g.push_back({Op::kLater, item_done});
        }
        s.push_back({Op::kLater, row_empty[Rows::buffer(n)]});
        math.push_back({Op::kArrive, row_empty[Rows::buffer(n)]});
        math.push_back({Op::kArrive, sched_empty[n % kRecords]});
    }
    m.roles.insert(m.roles.end(), {math, math, store, store, s, g});
    return m;
}

// visits[n][h]: bit i set where half h visits tile i of item n
template <uint32_t kTeams>
Model forward(const std::vector<int> &tiles, const std::vector<uint32_t> (&visits)[2]) {
    Model m;
    const int readers = 2 + 2 + kLoadWarps, parts = kLoadWarps / kTeams;
    const auto sched_full = m.add(kRecords, 1), sched_empty = m.add(kRecords, readers), row_full = m.add(2, parts),
               row_empty = m.add(2, 2 + 2), tile_full = m.add(kTileBufs, parts), tile_empty = m.add(kTileBufs, 2);
    loaders<kTeams>(m, tiles, sched_full, sched_empty, row_full, row_empty, tile_full, tile_empty, true);
    const uint32_t N = (uint32_t)tiles.size();
    for (int h = 0; h < 2; ++h) {
        const int s_full = m.add(1), s_free = m.add(1), p_full = m.add(1), pv_done = m.add(1);
        std::vector<Op> mma, soft;
        uint32_t c = 0, seen = 0;  // tiles, visits
        for (uint32_t n = 0; n <= N; ++n) {
            for (auto *o : {&mma, &soft}) o->push_back(wait(sched_full[n % kRecords], n / kRecords));
            mma.push_back({Op::kArrive, sched_empty[n % kRecords]});
            if (n == N) {
                soft.push_back({Op::kArrive, sched_empty[n % kRecords]});
                break;
            }
            for (auto *o : {&mma, &soft}) o->push_back({Op::kWait, row_full[Rows::buffer(n)], Rows::full_parity(n), n / 2 + 1});
            bool out = false;
            int in_unit = 0;
            for (int i = 0; i <= tiles[n]; ++i) {
                const bool visit = i < tiles[n] && (visits[h][n] >> i & 1);
                if (visit) mma.push_back({Op::kWait, tile_full[Tiles::buffer(c + i)], Tiles::full_parity(c + i), (c + i) / kTileBufs + 1});
                if (out) mma.push_back(wait(s_free, (int64_t)seen - 1));
                if (visit) mma.push_back({Op::kLater, s_full});
                if (out) {
                    mma.push_back(wait(p_full, (int64_t)seen - 1));
                    mma.push_back({Op::kLater, pv_done});
                    mma.push_back({Op::kLater, tile_empty[Tiles::buffer(c + i - 1)]});
                }
                if (!visit && i < tiles[n]) {
                    mma.push_back({Op::kWait, tile_full[Tiles::buffer(c + i)], Tiles::full_parity(c + i), (c + i) / kTileBufs + 1});
                    mma.push_back({Op::kArrive, tile_empty[Tiles::buffer(c + i)]});
                }
                if (visit) {
                    soft.push_back(wait(s_full, seen));
                    soft.push_back({Op::kArrive, s_free});
                    if (in_unit++ > 0) soft.push_back(wait(pv_done, (int64_t)seen - 1));
                    soft.push_back({Op::kArrive, p_full});
                    ++seen;
                }
                out = visit;
            }
            if (in_unit > 0) soft.push_back(wait(pv_done, (int64_t)seen - 1));
            c += tiles[n];
            mma.push_back({Op::kLater, row_empty[Rows::buffer(n)]});
            soft.push_back({Op::kArrive, row_empty[Rows::buffer(n)]});
            soft.push_back({Op::kArrive, sched_empty[n % kRecords]});
        }
        m.roles.push_back(mma);
        m.roles.push_back(soft);
    }
    return m;
}

// Random lists of up to 14 items of up to `most` tiles, half of them longest first: runs with an early wait in out[0], runs
// that stand still in out[1].
template <uint32_t kTeams>
void lists(bool bwd, int runs, int most, uint32_t seed, int *out) {
    std::mt19937 rng(seed);
    out[0] = out[1] = 0;
    for (int r = 0; r < runs; ++r) {
        std::vector<int> tiles(1 + rng() % 14);
        for (int &t : tiles) t = (int)(rng() % (most + 1));
        if (rng() % 2) std::sort(tiles.rbegin(), tiles.rend());
        std::vector<uint32_t> visits[2];
        for (auto &v : visits)
            for (size_t n = 0; n < tiles.size(); ++n) v.push_back(rng() % 4 ? (rng() % 2 ? ~0u : (uint32_t)rng()) : 0);
        Model m = bwd ? backward<kTeams>(tiles) : forward<kTeams>(tiles, visits);
        const int what = m.run(rng);
        if (what) ++out[what - 1];
    }
}

}  // namespace

extern "C" void as_built(int bwd, int runs, int most, unsigned seed, int *out) { lists<1>(bwd != 0, runs, most, seed, out); }
// loads by two teams of warps in turn
extern "C" void teams(int bwd, int runs, int most, unsigned seed, int *out) { lists<2>(bwd != 0, runs, most, seed, out); }
