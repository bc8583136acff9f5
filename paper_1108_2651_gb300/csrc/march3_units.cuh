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

// The time of a launch of the marching kernel and of a single step, measured on 22 grids from 32^3 to 192^3 and from 3 to
// 131072 planes, rows or columns (more: with walls, with sigma written, and for the adjoint).  Marching takes 2.2 to 2.6 us
// a plane of a wave of blocks (walls 3.0 to 3.4), a single step 27 ns a thousand elements of a plane, its rows' padding
// included (a warp takes 32 of a row whatever it holds), but no launch less than 4.1 us: 3 x 250 x 460 34.0 us a launch
// against three steps of 8.7 (walls 45.9, 11.1), 30 x 24 x 96 14.1 against 4.1, 48^3 14.5 against 6.1, 64^3 23.7 against 8.2
// (walls 32.5, 10.1), 80^3 30.0 against 16.4 (walls 40.3, 18.4), 192^3 318 against 180 (walls 398, 187).
inline double march3_us(const March3Plan &p, bool more) { return (double)p.planes * (more ? 3.35 : 2.4); }
inline double single3_us(double plane, bool more) {
    return std::max(4.1, (more ? 2. : 1.2) + plane * (more ? 27.5e-6 : 27e-6));
}

}  // namespace lbk
