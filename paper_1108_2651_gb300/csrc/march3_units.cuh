// The 3D marching kernel's blocks (march3d.cu): host code, plain C++.
#pragma once
#include <algorithm>
#include <vector>

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
// In a CUDA graph a marching launch takes 2.1 us more than in a stream and a single step 0.7 us less (64^3 8.6 us a step by
// marching against 7.5, 80^3 10.7 against 15.5).
inline double march3_us(const March3Plan &p, int nx, bool more) {
    const double plane = more ? 3.35 : 2.4;
    return (double)p.planes * (nx < 8 ? 1.65 * plane : plane);  // (460 x 250 x 3: 4.0 us a plane, walls 4.6)
}
inline double single3_us(double plane, bool more) {
    return std::max(4.1, (more ? 2. : 1.2) + plane * (more ? 27.5e-6 : 27e-6));
}

// What a handle's events (rowptr: those of row z ny + y before it) add to a launch of the marching kernel and to a single
// step, in us.  A warp of a block goes through every event of each of its two rows that has one in the tile's columns, at
// each of the K levels of a plane, while the block waits: 0.4 us a row and 0.09 us an event (64^3 with 16384 receivers at
// random 29.0 us a step against 8.2 without, 10.3 by single steps; with 1024 11.6 and 8.3; 3 x 250 x 460 with 16384 69.9
// and 16.5; 192^3 with 16384 139 and 184).  A single step has a warp a row: 0.15 us an event of the fullest row.
struct March3Events {
    double launch = 0., step = 0.;
};
inline March3Events march3_events_us(const March3Plan &p, int nx, int ny, int nz, int K, const std::vector<int> &rowptr) {
    March3Events us;
    struct Tile {      // of one plane
        double hits = 0.;  // rows that have an event in one tile's columns, if a row's events lie evenly
        int rows = 0, events = 0;
    };
    std::vector<Tile> row(p.nty);
    std::vector<double> sum((size_t)p.nty * (nz + 1), 0.);  // [row of tiles][planes before]
    int fullest = 0;
    auto start = [&](int t) { return (int)((long long)t * ny / p.nty); };
    for (int z = 0; z < nz; z++) {
        const int *r = rowptr.data() + (long long)z * ny;
        if (r[ny] == r[0]) {
            for (int t = 0; t < p.nty; t++) sum[(size_t)t * (nz + 1) + z + 1] = sum[(size_t)t * (nz + 1) + z];
            continue;
        }
        row.assign(p.nty, Tile());
        int t = 0, y0 = 0, y1 = start(1);  // the tile of y and its rows
        for (int y = 0; y < ny; y++) {
            if (y >= y1) {
                t++;
                y0 = y1;
                y1 = start(t + 1);
            }
            const int n = r[y + 1] - r[y];
            if (n == 0) continue;
            fullest = std::max(fullest, n);
            auto add = [&](Tile &a) {
                a.hits += std::min(1., n * 32. / nx);
                a.rows++;
                a.events += n;
            };
            add(row[t]);  // and the tiles that march it as one of their K - 1 rows at either side
            if (p.nty > 1 && y - y0 < K - 1) add(row[t > 0 ? t - 1 : p.nty - 1]);
            if (p.nty > 1 && y1 - y < K) add(row[t < p.nty - 1 ? t + 1 : 0]);
        }
        for (t = 0; t < p.nty; t++) {
            const Tile &a = row[t];
            const double most = a.hits < 1. ? a.hits : std::min(2., 1. + (a.hits - 1.) / 8.);  // of a warp's two rows
            sum[(size_t)t * (nz + 1) + z + 1] =
                sum[(size_t)t * (nz + 1) + z] + (a.rows ? most * (0.4 + 0.09 * a.events / a.rows) : 0.);
        }
    }
    double worst = 0., all = 0.;  // over the rows of tiles and the segments
    int len = 0;
    for (int k = 0; k < p.nseg; k++) {  // a segment's planes and the K - 1 at either end
        const int z0 = (int)((long long)k * nz / p.nseg), z1 = (int)((long long)(k + 1) * nz / p.nseg);
        len = std::max(len, z1 - z0);
        for (int t = 0; t < p.nty; t++) {
            const double *s = sum.data() + (size_t)t * (nz + 1);
            auto upto = [&](int z) {  // planes 0 .. z - 1, wrapped
                const int q = z >= 0 ? z / nz : -((-z + nz - 1) / nz);
                return q * s[nz] + s[z - q * nz];
            };
            const double v = upto(z1 + K - 1) - upto(z0 - (K - 1));
            worst = std::max(worst, v);
            all += v;
        }
    }
    // one wave waits for the worst block, the others take the mean
    const double waves = (double)p.planes / (len + 2 * (K - 1));
    us.launch = K * (worst + (waves - 1.) * all / ((double)p.nty * p.nseg));
    us.step = 0.15 * fullest;
    return us;
}

}  // namespace lbk
