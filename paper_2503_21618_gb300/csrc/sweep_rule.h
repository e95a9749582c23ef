// CTAs per SM of the exact level's sweep update (host code, no CUDA types).
#pragma once
#include <stdint.h>

namespace slrf {

// Three CTAs per SM or two, by the launch's number of tiles.  The launch ends
// with the CTAs that sweep the next diagonal blocks, which are faster beside one
// other CTA than beside two; three per SM pay where they fill the last of several
// waves (over three fifths of it), and where there are no more than two per SM
// anyway the larger shared-memory request of two only delays their start.  Cycle
// call, three against two per SM, by the number of tiles on 152 SMs: 112: 370 / 395
// us, 264: 711 / 721, 420: 870 / 803, 480: 1073 / 906, 684 (half of the last wave):
// 1147 / 1029, 840: 1232 / 1303, 1104: 1764 / 1724, 1224 (68 %): 1432 / 1533, 1368
// (full): 1626 / 1719, 2280 (full): 2595 / 2765.
inline bool sweep_three_per_sm(int sm_count, int64_t tiles) {
    const int64_t wave = 3 * (int64_t)sm_count;
    const int64_t last = tiles > 0 ? (tiles - 1) % wave + 1 : 0;   // tiles of the last wave; a full one counts as full
    return tiles <= 2 * (int64_t)sm_count || (tiles > wave && 5 * last > 3 * wave);
}

}  // namespace slrf
