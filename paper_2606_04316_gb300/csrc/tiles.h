// tiles.h -- the integral kernel's tile lists on the host: cutting a class's kept quartets
// into tiles, and the room such a list takes.  No CUDA calls, shared by the library and its
// CPU tests.
#pragma once

#include <algorithm>
#include <vector>

#include "plan.h"
#include "qdt_internal.cuh"

namespace qdt {

// Tiles of at most tile_kets() kets of one bucket per bra pair (list: shell pair at
// each ket position); with `split`, positions [0, split) and [split, prefix) are tiled
// apart, the second set in plain FP32 and after all tiles of the first for these bra pairs: the phases of both forms together are more code than the
// instruction caches hold (interleaved, the integrals of a 40-centre chain took 131.1 ms
// instead of 125.2, of a 24-centre chain 172.6 instead of 169.0).
inline void build_tiles(const PairClass &pc, const std::vector<int> &bras, const std::vector<int> &prefix,
                        const KetBuckets &kb, const BucketCounts &below, const std::vector<int> &list, bool gauge,
                        const EriLaunch &how, int req, std::vector<EriTask> &out, const std::vector<int> *split = nullptr) {
    for (int kind = 0; kind < (split ? 2 : 1); ++kind)
        for (int sp : bras)
            for (int b = 0; b + 1 < (int)kb.first.size(); ++b) {
                const PairDev &CD = pc.h_pairs[list[kb.pos[kb.first[b]]]];
                const int kets = tile_kets(pc.h_pairs[sp], CD, gauge, how.budget, how.kets);
                const int f = kb.first[b], pre = f + below(b, prefix[sp]);
                const int mid = split ? f + below(b, (*split)[sp]) : pre, end = kind ? pre : mid;
                for (int q = kind ? mid : f; q < end; q += kets)
                    out.push_back({sp, q, std::min(end, q + kets), req, kind});
            }
}

// Counts shell pair `id` of a class into its kinds (pairs of one kind share their FuncPair table).
inline void count_kind(PairClass &pc, int id) {
    const PairDev &p = pc.h_pairs[id];
    for (PairClass::Kind &k : pc.kinds)
        if (pc.h_pairs[k.most].fpoff == p.fpoff) {
            ++k.pairs;
            k.npp += p.npp;
            if (p.npp > pc.h_pairs[k.most].npp) k.most = id;
            return;
        }
    pc.kinds.push_back({1, id, p.npp});
}

// Mean cost of a class's quartets, over pairs of kinds with their mean numbers of primitive
// pairs: a few hundred evaluations where a basis of long contractions has a thousand buckets,
// whose pairs took 14 ms of host time in every row batch.  (The cost is bilinear in the numbers
// but for the choice of the orientation.)
inline double mean_quartet_cost(const PairClass &pc, bool gauge) {
    double sum = 0.0, weight = 0.0;
    for (const PairClass::Kind &a : pc.kinds)
        for (const PairClass::Kind &c : pc.kinds) {
            const double w = (double)a.pairs * c.pairs;
            sum += w * quartet_cost_of<double>(pc.h_pairs[a.most], (double)a.npp / a.pairs, pc.h_pairs[c.most],
                                               (double)c.npp / c.pairs, gauge);
            weight += w;
        }
    return weight > 0.0 ? sum / weight : 0.0;
}

// Smallest tile that tile_kets() gives any two pairs of the class: the cost grows with the primitive
// pairs, so the longest pair of each kind is enough.
inline int smallest_tile(const PairClass &pc, bool gauge, const EriLaunch &how) {
    int least = how.kets;
    for (const PairClass::Kind &a : pc.kinds)
        for (const PairClass::Kind &c : pc.kinds)
            least = std::min(least, tile_kets(pc.h_pairs[a.most], pc.h_pairs[c.most], gauge, how.budget, how.kets));
    return least;
}

// Room that the tiles of these bra pairs take at most (nbucket: buckets of the ket list; one or
// two kinds of tile): full tiles of the smallest size under this very launch shape and, for every
// bucket of a bra pair, a part tile of each kind.
inline long long tile_bound(const PairClass &pc, const std::vector<int> &bras, const std::vector<int> &prefix,
                            int nbucket, bool gauge, const EriLaunch &how) {
    const int least = smallest_tile(pc, gauge, how);
    long long most = 0;
    for (int sp : bras) most += prefix[sp] / least + std::min<long long>(2LL * nbucket, prefix[sp]);
    return most;
}

}  // namespace qdt
