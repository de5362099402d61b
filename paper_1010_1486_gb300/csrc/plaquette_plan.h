// plaquette_plan.h -- how the plaquette kernel's work is cut.  Host code alone.
#pragma once

#include <algorithm>

namespace su2 {

constexpr int kPlaqPairs = 384;         // pairs of sites (2 j, 2 j + 1) per block
constexpr double kPlaqItemSteps = 0.2;  // steps that an item's start costs

// The work is pair blocks x chunks of t_chunk time slices, in that order; one
// block per SM takes every grid-th item.
struct PlaquettePlan {
    int pair_blocks, t_chunk, items, grid;
};

// The chunk length with which the block that has most to do ends first.  One
// item per block and the time extent in as many chunks as fill the SMs (rounded
// down) left up to half of them idle between the extents that happen to fit:
// 40^4 84 blocks, 50^4 163, a second wave of eleven.  us per call, the kernel
// of one site per thread / one item per block / this: 40^4 63 / 76 / 55, 44^4
// 79 / 84 / 68, 48^4 100 / 91 / 90, 50^4 116 / 171 / 106, 56^4 168 / 190 / 154,
// 64^4 265 / 311 / 240, 24^4 27 / 21 / 21.  (With 0.5, 1 or 2 steps for the start
// of an item 46^4, 50^4, 54^4 or 60^4 take 4 to 10% longer.)
inline PlaquettePlan plaquette_plan(int vs, int nt, int sms)
{
    PlaquettePlan p = {};
    p.pair_blocks = (vs / 2 + kPlaqPairs - 1) / kPlaqPairs;
    p.t_chunk = nt;
    p.items = p.pair_blocks;
    double best = (double)((p.items + sms - 1) / sms) * (nt + kPlaqItemSteps);
    for (int rounds = 1; rounds <= 16; ++rounds) {
        const int chunks = std::min(nt, rounds * sms / p.pair_blocks);
        if (chunks < 1) continue;
        const int t_chunk = (nt + chunks - 1) / chunks, items = p.pair_blocks * ((nt + t_chunk - 1) / t_chunk);
        const double cost = (double)((items + sms - 1) / sms) * (t_chunk + kPlaqItemSteps);
        if (cost < best) {
            best = cost;
            p.t_chunk = t_chunk;
            p.items = items;
        }
    }
    p.grid = std::min(p.items, sms);
    return p;
}

}  // namespace su2
