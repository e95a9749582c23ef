// CTAs per SM of the exact level's sweep update (host code, no CUDA types).
#pragma once
#include <stdint.h>

namespace slrf {

// Three CTAs per SM or two, by the launch's number of tiles.  The launch ends
// with the CTAs that sweep the next diagonal blocks, which are faster beside one
// other CTA than beside two.  That counts where a launch is one or two waves of
// three per SM long; in the second of two, three per SM pay where they fill over
// three fifths of it, and up to two CTAs per SM it makes no difference.  Cycle
// call on 152 SMs, three against two per SM, by the number of tiles: 112: 292 / 293
// us, 264: 488 / 489, 420: 692 / 619, 480: 735 / 688, 612: 854 / 855, 684: 960 / 935,
// 760: 1050 / 1088, 840: 1171 / 1214, 918: 1130 / 1179, 1104: 1641 / 1715, 1368: 1594 /
// 1664, 2280: 2605 / 2824.
inline bool sweep_three_per_sm(int sm_count, int64_t tiles) {
    const int64_t wave = 3 * (int64_t)sm_count;
    return tiles <= 2 * (int64_t)sm_count || 5 * tiles > 8 * wave;
}

}  // namespace slrf
