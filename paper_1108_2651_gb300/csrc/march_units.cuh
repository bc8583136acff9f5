// The 2D marching kernel's units (march.cuh) and what a handle's events cost in them (host code; plain C++ but for
// march_cut and march_row, which the kernel uses too).
#pragma once
#include <algorithm>
#include <vector>

#ifdef __CUDACC__
#define MARCH_HD __host__ __device__ __forceinline__
#else
#define MARCH_HD inline
#endif

namespace lbk {

// A unit's column and row ranges: whole chunks of 4 columns and rows, evenly.
MARCH_HD int march_cut(int k, int n, int of) { return (int)((long long)k * of / n); }
// The first row of segment k of n, of ny rows, the first and the last segment of he rows (0: as the others).
MARCH_HD int march_row(int k, int n, int ny, int he) {
    if (he == 0 || k == 0 || k == n) return k == n ? ny : march_cut(k, n, ny);
    return he + march_cut(k - 1, n - 2, ny - 2 * he);
}

constexpr int MARCH_RECORDS = 32;  // sources and receivers that a unit lists in shared memory

// The units of a launch of K steps with H halo columns: nstrips strips of columns by nseg segments of rows, of which
// the first nl and last nr strips (walled columns or layers) have nsegx, and the first and last segment of the others
// he rows (0: as the rest).
struct MarchUnits {
    int K = 0, H = 0, nstrips = 0, nseg = 0, nl = 0, nr = 0, nsegx = 0, he = 0;
    bool walled(int strip) const { return strip < nl || strip >= nstrips - nr; }
    int segs(int strip) const { return walled(strip) ? nsegx : nseg; }
    int row0(int strip, int k, int ny) const { return march_row(k, segs(strip), ny, walled(strip) ? 0 : he); }
};

struct MarchEvent {
    int row, x;
    bool source;
};
struct MarchEventCost {
    double visits = 0.;  // the most events a unit looks up one after another, a step (a source counts 2.5: its amplitude)
    int row = 0;         // the most events of a row
};

// What the marching kernel's units spend on these events on a grid of nx x ny with event buckets of `bucket` columns.  A
// unit lists up to 32 records; a unit with more, or with two sources on a site, looks up at every level every event of
// every row that has one in a bucket of its columns.  (The order of ev is lost.)
inline MarchEventCost march_event_cost(const MarchUnits &u, int nx, int ny, int bucket, std::vector<MarchEvent> &ev) {
    MarchEventCost c;
    const int nchunk = (nx + 3) / 4;
    std::vector<unsigned long long> mask(ny, 0);
    std::vector<double> weight(ny, 0.);
    std::vector<int> count(ny, 0);
    for (const MarchEvent &e : ev) {
        mask[e.row] |= 1ull << (e.x / bucket);
        weight[e.row] += e.source ? 2.5 : 1.;
        c.row = std::max(c.row, ++count[e.row]);
    }
    std::vector<int> col(u.nstrips + 1, nx), first(u.nstrips + 1, 0);  // a strip's first column and first unit
    for (int s = 0; s < u.nstrips; s++) {
        col[s] = 4 * march_cut(s, u.nstrips, nchunk);
        first[s + 1] = first[s] + u.segs(s);
    }
    std::vector<int> rows[2];  // the first rows of the segments of the strips without and with walls, and ny
    for (int k = 0; k <= u.nseg; k++) rows[0].push_back(march_row(k, u.nseg, ny, u.he));
    for (int k = 0; k <= u.nsegx; k++) rows[1].push_back(u.nsegx ? march_row(k, u.nsegx, ny, 0) : ny);
    auto last_from = [](const std::vector<int> &v, int at) {  // the last of them that begins at or before `at`
        const int n = (int)v.size() - 1;
        int k = std::min((int)((double)at * n / v[n]), n - 1);  // (cut about evenly)
        while (k + 1 < n && v[k + 1] <= at) k++;
        while (k > 0 && v[k] > at) k--;
        return k;
    };
    std::vector<int> rec(first[u.nstrips], 0);
    const int out = u.K - 1;  // rows that a unit marches before and after its own
    const auto sources = std::partition(ev.begin(), ev.end(), [](const MarchEvent &e) { return !e.source; });
    for (auto e = ev.begin(); e != sources; ++e) {
        const int s = last_from(col, e->x);
        rec[first[s] + last_from(rows[u.walled(s)], e->row)]++;
    }
    std::sort(sources, ev.end(), [](const MarchEvent &a, const MarchEvent &b) {
        return a.row != b.row ? a.row < b.row : a.x < b.x;
    });
    for (auto e = sources; e != ev.end(); ++e) {
        const bool twice = e != sources && (e - 1)->row == e->row && (e - 1)->x == e->x;
        const int own = last_from(col, e->x);
        // strips (56 to 112 columns wide, or one) whose 128 columns hold the source, once or, on a narrow grid, several times
        for (int d = -std::min(3, (u.nstrips - 1) / 2); d <= std::min(3, u.nstrips / 2); d++) {
            const int s = (own + d + u.nstrips) % u.nstrips;
            int dx = (e->x - (col[s] - u.H)) % nx;
            dx += dx < 0 ? nx : 0;
            const int copies = dx < 128 ? (127 - dx) / nx + 1 : 0;
            if (!copies) continue;
            const std::vector<int> &r = rows[u.walled(s)];
            for (int y = e->row - (out + ny - 1) / ny * ny; y < ny + out; y += ny)  // the rows that wrap to it
                for (int k = last_from(r, std::min(std::max(y - out, 0), ny - 1)); k < u.segs(s) && r[k] - out <= y; k++)
                    if (y < r[k + 1] + out) rec[first[s] + k] += twice ? MARCH_RECORDS + 1 : copies;
        }
    }
    for (int s = 0; s < u.nstrips; s++) {
        const std::vector<int> &r = rows[u.walled(s)];
        unsigned long long cols = 0;  // the buckets of the strip's columns
        bool known = false;
        for (int k = 0; k < u.segs(s); k++) {
            if (rec[first[s] + k] <= MARCH_RECORDS) continue;
            for (int j = 0; j < 128 && !known; j++) {
                const int x = (col[s] - u.H + j) % nx;
                cols |= 1ull << ((x < 0 ? x + nx : x) / bucket);
            }
            known = true;
            double v = 0.;
            int row = (((r[k] - out) % ny) + ny) % ny;
            for (int y = r[k] - out; y < r[k + 1] + out; y++, row = row + 1 == ny ? 0 : row + 1)
                if (mask[row] & cols) v += weight[row];
            c.visits = std::max(c.visits, v);
        }
    }
    return c;
}

}  // namespace lbk
