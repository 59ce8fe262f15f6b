// Output slices of a launch of the streaming apply kernel: how many items (units) a tile gives, chosen on the host in front of the launch.
#pragma once
#include <stdint.h>

#include <algorithm>

#include "molora.h"

namespace molora {

// Chunks of d_in and d_out of the launch's projections, heaviest projection first.
struct SliceShapes {
    int P;
    int in[MOLORA_MAX_PROJECTIONS], out[MOLORA_MAX_PROJECTIONS];
};

// One unit per projection to start with; while `most` units allow it, the widest is split once more.  Projection p owns units
// [ustart[p], ustart[p + 1]) of och[p] chunks of d_out each.  Returns the number of units.
inline int slice_outputs(const SliceShapes& sh, int64_t most, int32_t* och, int32_t* ustart)
{
    int slices[MOLORA_MAX_PROJECTIONS], total = sh.P;
    for (int i = 0; i < sh.P; ++i) {
        och[i] = sh.out[i];
        slices[i] = 1;
    }
    for (; total + 1 <= most; ++total) {
        int widest = 0;
        for (int i = 1; i < sh.P; ++i)
            if (och[i] > och[widest]) widest = i;
        if (och[widest] <= 1) break;
        ++slices[widest];
        och[widest] = (sh.out[widest] + slices[widest] - 1) / slices[widest];
    }
    ustart[0] = 0;
    for (int i = 0; i < sh.P; ++i) ustart[i + 1] = ustart[i] + (sh.out[i] + och[i] - 1) / och[i];
    return ustart[sh.P];
}

// Work of the busiest cluster when `tiles` items of every unit are dealt to the clusters, from the front and from the back in turn.  The
// items of a unit cost the same, so they are added as ranges of clusters, one per round, and the clusters are walked once.
constexpr int kSliceMaxClusters = 256;
constexpr int kShrinkJobCost = 13, kExpandJobCost = 20, kItemCost = 8;      // see balanced_units
inline int busiest_cluster(const SliceShapes& sh, const int32_t* och, const int32_t* ustart, int clusters, int tiles)
{
    int step[kSliceMaxClusters + 1] = {};              // load[c] = step[0] + ... + step[c]
    int round = 0, at = 0;                             // of the next item: position in its round
    for (int p = 0; p < sh.P; ++p)
        for (int u = ustart[p]; u < ustart[p + 1]; ++u) {
            const int chunks = std::min<int>(och[p], sh.out[p] - (u - ustart[p]) * och[p]);
            const int cost = kShrinkJobCost * sh.in[p] + kExpandJobCost * chunks + kItemCost;
            for (int left = tiles; left > 0;) {
                const int n = std::min(left, clusters - at);
                const int lo = (round & 1) ? clusters - at - n : at;
                step[lo] += cost;
                step[lo + n] -= cost;
                left -= n;
                at += n;
                if (at == clusters) at = 0, ++round;
            }
        }
    int load = 0, longest = 0;
    for (int c = 0; c < clusters; ++c) longest = std::max(longest, load += step[c]);
    return longest;
}

// Output slices of calls whose items no longer fit one wave (one CTA per item): the launch lasts as long as its busiest CTA, and a
// gate or up projection in a layer is six expand jobs behind two shrinks while the average CTA has five jobs.  Cutting it in two costs
// two more shrinks and evens that out.  The dealing of the items is followed for the tiles that are expected, with up to four cuts; a
// shrink job counts 0.65 of an expand job (measured in place at rank 16: 1240 and 1900 cycles).  256 tokens of 8 adapters, sixteen layers
// 2048 wide: 207 us without cuts, 186 with.
// How many tiles there are depends on the load, which the host does not know, so a cut must not lengthen the launch of an evenly spread one
// (equal_tiles) either: of 32 adapters 40 tokens are expected to meet 20 and may meet all, and the cuts for 20 tiles made a layer 3072 wide
// 23.3 us where none take 18.3 (36 tokens, 2560 wide 21.1 / 16.8; rank 64, 44 tokens, 512 wide 17.8 / 15.4).
// The costs are those of rank 16; layers and attention projections of all ranks, 16 to 1200 tokens, us with cuts / without, where the
// rule cuts: rank 16 0.87 to 1.0, rank 32 0.91 to 1.03, rank 64 0.90 to 1.0 of the time.  Returns the number of units.
inline int balanced_units(const SliceShapes& sh, int clusters, int tiles, int equal_tiles, int32_t* och, int32_t* ustart)
{
    constexpr int kCuts = 4;
    int best_units = sh.P, best = 0, best_equal = 0;
    for (int most = sh.P; most <= sh.P + kCuts; ++most) {
        if (slice_outputs(sh, most, och, ustart) < most) break;
        const int longest = busiest_cluster(sh, och, ustart, clusters, tiles);
        if (most > sh.P && (int64_t)longest * 100 >= (int64_t)best * 97) continue;
        const int equal = equal_tiles == tiles ? longest : busiest_cluster(sh, och, ustart, clusters, equal_tiles);
        if (most > sh.P && equal > best_equal) continue;
        best = longest;
        best_equal = equal;
        best_units = most;
    }
    return slice_outputs(sh, best_units, och, ustart);
}

}  // namespace molora
