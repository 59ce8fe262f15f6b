// CTAs per tile of a launch of the tcgen05 apply kernel, chosen on the host in front of the launch.
#pragma once
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "molora.h"

namespace molora {

struct UmmaPlan {
    int split;       // CTAs per tile (cluster size)
    int tile_rows;   // positions per tile
};

// Tiles per projection of N tokens of C adapters: of an evenly spread load, whose segments all round up together, and of an uneven one,
// whose segments end in half a tile on average with a spread of sqrt(C / 12) over C random remainders.
struct UmmaTiles {
    int64_t equal, uneven;
};
inline UmmaTiles umma_tiles(int64_t N, int32_t C, int rows)
{
    auto up = [](int64_t a, int64_t b) { return (a + b - 1) / b; };
    return {(int64_t)C * up(up(N, C), rows), std::max<int64_t>(C, up(N, rows) + (int64_t)(C / 2.0 + std::sqrt(C / 12.0)))};
}

// Tiles are 128 rows, so small calls have too few of them for 148 SMs; a tile can be split over a cluster (up to 4 CTAs; up to 8 at
// rank 64).  Picks the split with the smallest estimated time, in microseconds, from a model fitted to one-projection 4096 -> 4096 calls
// at rank 64 (64 ... 4096 tokens, every split, graph replay): a wave of resident clusters costs a fixed 9 us (launch, tile look-up, first
// arrival, last stores), 3 us more for the exchange of the partial T tiles, and 0.40 us per 64-column chunk a CTA walks (shrink
// chunks + expand chunks divided by the split); shorter tiles make a chunk only a little cheaper (the gathers are bound by requests in
// flight, not bytes).
// Which load there is the host does not know, and the errors do not cost the same: a tile more than the resident clusters makes a second
// wave.  So a split is charged what it takes under both, the worse one in full and half of their mean on top.  Of 2160 calls (ranks 32 and
// 64; one, two, four and seven projections 1024 - 4096 wide, 600 - 8000 tokens, 2 - 16 adapters, three loads) 29 shapes choose another
// split than for the larger number of tiles alone, from 16 % faster to 4 % slower, 3 % faster in the mean; none is slower than with
// N / 128 + C / 2 tiles, which the kernel before had (1700 tokens of 16 adapters, four projections 2048 wide: one CTA a tile 32.7 us,
// two 25.3; 3000 of 16, 1024 -> 1024: four 20.3, three 17.3; the worst of it: 1300 of 4, four 4096 wide: two 33.4, three 34.3).
//   chunks    64-column chunks that a tile of each of the nproj projections walks (d_in + d_out); min_kx: least of d_in
//   resident  clusters of that many CTAs that are resident at once
template <typename Resident>
UmmaPlan choose_umma_split(const double* chunks, int nproj, int min_kx, int64_t N, int32_t C, int max_split, int sms, Resident resident)
{
    // Estimated time of the launch: the CTAs are dispatched heaviest projection first onto the resident clusters, so the
    // launch lasts as long as its heaviest tile or as the whole work spread over the cluster slots (plus a quarter of a
    // light tile of imbalance), whichever is longer; with equal tiles it is whole waves.
    auto cost_of = [&](int64_t tiles, int rows, int split, bool& one_wave) {
        const int slots = resident(split);
        // (a chunk costs up to 1.4 times as much once every SM streams: 35 GB/s per SM instead of ~50)
        const double load = std::min(1.0, (double)(tiles * nproj * split) / sms);
        const double fixed = 9.0 + (split > 1 ? 3.0 : 0.0);
        const double per_chunk = 0.40 * (1.0 + 0.4 * load * load) * (0.7 + 0.3 * rows / 128.0) / split;
        double cmax = 0.0, cmin = 1e30, total = 0.0;
        for (int i = 0; i < nproj; ++i) {
            const double c = fixed + per_chunk * chunks[i];
            cmax = std::max(cmax, c);
            cmin = std::min(cmin, c);
            total += c * (double)tiles;
        }
        if (tiles * nproj * 1.1 <= slots) return cmax;       // (margin: the tile count is an estimate)
        one_wave = false;
        // (a wave that is almost full takes longer: 25 tiles on the 26 clusters of five that fit 21.5 us, on clusters of four 18.3)
        if (cmax - cmin < 1e-9) return cmax * (1.08 * (double)((tiles * nproj + slots - 1) / slots));
        return std::max(cmax, total / slots + 0.25 * cmin);
    };
    auto cost_for = [&](int rows, int split, bool& one_wave) {
        const UmmaTiles t = umma_tiles(N, C, rows);
        one_wave = true;
        const double a = cost_of(t.equal, rows, split, one_wave), b = cost_of(t.uneven, rows, split, one_wave);
        return std::max(a, b) + 0.25 * (a + b);
    };
    UmmaPlan best = {1, 128};
    if (nproj > 0) {
        double best_cost = 1e30;
        bool best_one_wave = false;
        for (int split = 1; split <= max_split; ++split) {    // cluster sizes need not be powers of two
            bool one_wave;
            const double cost = cost_for(128, split, one_wave);
            if (cost < best_cost - 1e-9) { best_cost = cost; best_one_wave = one_wave; best = {split, 128}; }
        }
        // A call that does not even fill one wave can use shorter tiles (the MMA tile keeps 128 lanes, the extra
        // lanes idle) to put more SMs to work, as long as everything still fits in one wave.
        const UmmaTiles t = umma_tiles(N, C, 128);
        if (best_one_wave && std::max(t.equal, t.uneven) * nproj * best.split < 0.85 * sms) {
            for (int rows = 96; rows >= 64; rows -= 32)
                for (int split = 1; split <= max_split; ++split) {
                    bool one_wave;
                    const double cost = cost_for(rows, split, one_wave);
                    if (one_wave && cost < best_cost - 1e-9) { best_cost = cost; best = {split, rows}; }
                }
        }
    }
    while (best.split > 1 && min_kx / best.split < 4) --best.split;   // keep at least four chunks of d_in per CTA
    return best;
}

}  // namespace molora
