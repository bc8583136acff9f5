// The 3D marching kernel's blocks (march3d.cu): host code, plain C++.
#pragma once
#include <algorithm>

namespace lbk {

constexpr int M3_PLANES = 512;  // the most planes a block marches

// Tiles of columns, segments of planes, and the planes that the waves of blocks march one after another.
struct March3Plan {
    int ntx = 1, nty = 1, nseg = 1;
    long long planes = 0;
};

// K steps, tiles of 32 x TY columns, `wave` blocks at a time: the segments for which the waves of blocks times the planes a
// block marches (its K - 1 at either end included) are the fewest.  More segments within the same waves only shorten them,
// so one number of segments a wave count is looked at, and w waves cost at least w (2 K - 1): a few hundred tries at most
// (trying every number of segments took a call on 131072 x 1 x 4 sites 450 us of host time).
inline March3Plan march3_plan(int nx, int ny, int nz, int K, int TY, int wave) {
    const int halo = 2 * (K - 1), wx = 32 - halo, wy = TY - halo;
    March3Plan p;
    p.ntx = (nx + wx - 1) / wx;
    p.nty = (ny + wy - 1) / wy;
    const long long tiles = (long long)p.ntx * p.nty;
    const long long least = (nz - 1) / (M3_PLANES - 2 * K) + 1;
    long long best = -1;
    for (long long w = (tiles * least + wave - 1) / wave; best < 0 || w * (halo + 1) < best; w++) {
        const long long most = std::min<long long>(nz, w * wave / tiles);  // segments that w waves hold
        if (most >= least) {
            const long long len = (nz + most - 1) / most, n = (nz + len - 1) / len;
            const long long cost = (tiles * n + wave - 1) / wave * (len + halo);
            if (best < 0 || cost < best) {
                best = cost;
                p.nseg = (int)n;
            }
        }
        if (most == nz) break;
    }
    p.planes = best;
    return p;
}

}  // namespace lbk
