// Where the transposes of a specialised pass (tile_jit.cpp) need the CTA's warps
// to meet.
#pragma once

#include <vector>

#include "tiled.h"

namespace qsim {

// How the transpose into each stage synchronises. A transpose between stages
// with the same warp bits, none of them among the swizzled low position bits,
// stays inside each warp's own positions (the swizzle maps the positions with
// given warp bits to themselves). A transpose that is not local, or is local in
// other positions, waits for the CTA first if a local one came before it: in the
// loop over tiles the pass's last transpose comes before its first. (The FMA
// pipe and shared memory take turns where a CTA's warps move together: a stage
// took their sum, 2400 cycles a tile, with 2 CTAs per SM. Random layers n = 28
// complex64, 27 of 83 transposes local: 25.0 -> 24.5 ms; energy and gradient at
// n = 18, 64 members 3.08 -> 2.98 ms. Tiles of 2^12 in CTAs of 4 warps, 4 per SM,
// run a pass 13% faster but need 13 passes for 11: 25.5 ms.)
constexpr char kSyncLocal = 1, kSyncBefore = 2;
template <typename R> std::vector<char> transpose_sync(const TileParams<R> &P) {
    constexpr int WB = TileCfg<R>::WB;
    std::vector<char> out(P.n_stages, 0);
    auto warps = [&](int s) {
        int w = 0;
        for (int i = 0; i < WB; ++i) w |= 1 << P.st[s].wloc[i];
        return w;
    };
    int open = 0;  // warp bits of the local transposes since the CTA last met (0: none)
    for (int round = 0; round < 2; ++round)
        for (int s = 1; s < P.n_stages; ++s) {
            const int w = warps(s);
            const bool local = w == warps(s - 1) && (w & ((1 << swizzle_low_bits<R>()) - 1)) == 0;
            out[s] = (local ? kSyncLocal : 0) | (open != 0 && !(local && open == w) ? kSyncBefore : 0);
            open = local ? w : 0;
        }
    return out;
}

}  // namespace qsim
