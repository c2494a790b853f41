// CPU check of the integral kernel's tile lists (tiles.h, plan.h) on seeded random
// classes, from bases of cheap quartets (few kinds, long prefixes: the largest tiles) to
// mixed ones: the buckets group a ket list, the tiles of a bra pair cover each of its kept
// kets once, within one bucket and the launch shape's sizes, and the list's room
// (tile_bound) holds them for every shape a launch may take; the mean cost and the smallest
// tile of a class, taken over its kinds, agree with those over all its buckets.
#include <algorithm>
#include <cstdio>
#include <random>

#include "tiles.h"

int main() {
    using namespace qdt;
    int fails = 0;
    long long full = 0;               // lists that need more than half their room
    for (int seed = 1; seed <= 60; ++seed) {
        std::mt19937_64 rng(seed);
        const int nsp = 40 + (int)(rng() % (seed % 3 ? 300 : 2500)), nbk = 1 + (int)(rng() % (seed % 2 ? 6 : 80));
        const bool gauge = rng() % 2 != 0;
        PairClass pc;
        pc.nsp = nsp;
        std::vector<PairDev> kind(nbk);           // bucket by bucket; every third starts a kind
        for (int b = 0; b < nbk; ++b) {
            PairDev &k = kind[b];
            if (b % 3) {
                k = kind[b - 1];
                k.npp = k.npp % 12 + 1;
                continue;
            }
            k = PairDev{};
            k.fpoff = b;
            k.Lab = seed % 4 == 1 ? 0 : (int)(rng() % 5);
            k.npp = seed % 4 == 1 ? 1 : 1 + (int)(rng() % 9);
            k.nfp = 1 + (int)(rng() % (seed % 4 == 1 ? 2 : 18));
            k.nbox = k.nfp * (1 + (int)(rng() % 9));
        }
        std::vector<int> of(nbk, -1);
        for (int i = 0; i < nsp; ++i) {
            const int k = (int)(rng() % nbk);
            if (of[k] < 0) {
                of[k] = (int)pc.bucket_rep.size();
                pc.bucket_rep.push_back(i);
            }
            pc.h_pairs.push_back(kind[k]);
            pc.h_bucket.push_back(of[k]);
            count_kind(pc, i);
        }
        const int nbucket = (int)pc.bucket_rep.size();
        // a ket list: the class in random order, or (row batches) part of it
        std::vector<int> list(nsp);
        for (int i = 0; i < nsp; ++i) list[i] = i;
        std::shuffle(list.begin(), list.end(), rng);
        if (seed % 5 == 0) list.resize(nsp - nsp / 3);
        const KetBuckets kb = ket_buckets(list, pc.h_bucket, nbucket);
        const BucketCounts below(kb);
        const int n = (int)list.size(), nb = (int)kb.first.size() - 1;
        if ((int)kb.pos.size() != n || kb.first.back() != n) { std::printf("seed %d: positions lost\n", seed); ++fails; }
        for (int b = 0; b < nb; ++b)
            for (int i = kb.first[b]; i < kb.first[b + 1]; ++i)
                if (pc.h_bucket[list[kb.pos[i]]] != pc.h_bucket[list[kb.pos[kb.first[b]]]] ||
                    (i > kb.first[b] && kb.pos[i] <= kb.pos[i - 1])) {
                    std::printf("seed %d: bucket %d\n", seed, b);
                    ++fails;
                }
        std::vector<int> bras, prefix(nsp), split(nsp);
        for (int i = 0; i < nsp; ++i) {
            prefix[i] = rng() % 7 == 0 ? (int)(rng() % (n + 1)) : n;
            split[i] = rng() % 3 == 0 ? prefix[i] : (int)(rng() % (prefix[i] + 1));
            if (rng() % 8 == 0 || nsp < 400) bras.push_back(i);
        }
        long long mean = 0;
        for (int i : pc.bucket_rep)
            for (int j : pc.bucket_rep) mean += quartet_cost(pc.h_pairs[i], pc.h_pairs[j], gauge);
        mean /= (long long)nbucket * nbucket;
        // the sums over kinds against all pairs of buckets: the mean is exact but for the choice of
        // the orientation, for which a mean takes one and every bucket its own
        double sum = 0.0;
        for (int i = 0; i < nsp; ++i)
            for (int j : pc.bucket_rep)
                sum += (double)quartet_cost(pc.h_pairs[i], pc.h_pairs[j], gauge) *
                       (double)std::count(pc.h_bucket.begin(), pc.h_bucket.end(), pc.h_bucket[j]);
        sum /= (double)nsp * nsp;
        const double by_kind = mean_quartet_cost(pc, gauge);
        if (by_kind < sum * (1.0 - 1e-9) || by_kind > 2.0 * sum) {
            std::printf("seed %d: mean cost %.6e by kinds, %.6e\n", seed, by_kind, sum);
            ++fails;
        }
        for (long long budget : {0LL, 1LL, mean, 12 * mean, 200 * mean}) {
            EriLaunch how;
            how.budget = budget;
            int least = how.kets;
            for (int i : pc.bucket_rep)
                for (int j : pc.bucket_rep)
                    least = std::min(least, tile_kets(pc.h_pairs[i], pc.h_pairs[j], gauge, budget, how.kets));
            if (smallest_tile(pc, gauge, how) != least) { std::printf("seed %d: smallest tile\n", seed); ++fails; }
        }
        for (int kets : {1, 8, 16, kMaxTileKets})
            for (long long budget : {0LL, 1LL, mean, 3 * mean, 12 * mean, 200 * mean})
                for (int form = 0; form < 2; ++form) {
                    EriLaunch how;
                    how.kets = kets;
                    how.budget = budget;
                    std::vector<EriTask> t;
                    build_tiles(pc, bras, prefix, kb, below, list, gauge, how, 3, t, form ? &split : nullptr);
                    const long long room = tile_bound(pc, bras, prefix, nb, gauge, how);
                    if ((long long)t.size() > room) {
                        std::printf("seed %d: kets %d, budget %lld: %zu tiles, room for %lld\n", seed, kets, budget, t.size(), room);
                        ++fails;
                    }
                    full += 2 * (long long)t.size() > room;
                    std::vector<long long> got(nsp, 0);
                    std::vector<char> seen((size_t)nsp * n, 0);
                    int last = 0;
                    for (const EriTask &e : t) {
                        bool ok = e.req == 3 && e.k1 > e.k0 && e.k1 - e.k0 <= kets && e.f32 >= last && (form || !e.f32);
                        last = e.f32;
                        for (int i = e.k0; ok && i < e.k1; ++i) {
                            const int p = kb.pos[i];
                            char &s = seen[(size_t)e.bra_sp * n + p];
                            ok = p < prefix[e.bra_sp] && !s && (e.f32 != 0) == (form && p >= split[e.bra_sp]) &&
                                 pc.h_bucket[list[p]] == pc.h_bucket[list[kb.pos[e.k0]]];
                            s = 1;
                        }
                        got[e.bra_sp] += e.k1 - e.k0;
                        if (!ok && fails < 20) { std::printf("seed %d: a tile of bra pair %d\n", seed, e.bra_sp); ++fails; }
                    }
                    for (int sp : bras)
                        if (got[sp] != prefix[sp] && fails < 20) { std::printf("seed %d: kets of bra pair %d\n", seed, sp); ++fails; }
                }
    }
    if (full == 0) { std::printf("no list comes near its room\n"); ++fails; }
    std::printf(fails ? "FAILED %d\n" : "ok\n", fails);
    return fails ? 1 : 0;
}
