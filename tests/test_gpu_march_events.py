"""Sources and receivers that crowd a unit of the 2D marching kernel: the host's count of what they cost, the bits of the
rows that look events up one by one, and the rule that leaves crowded grids to launches of two steps."""
import os
import subprocess

import numpy as np
import pytest

from paper_1108_2651_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1108_2651_gb300", "csrc")

# march_event_cost against a count over every unit, row and event
HARNESS = r"""
#include "march_units.cuh"
#include <random>
using namespace lbk;
int main() {
    std::mt19937 gen(1);
    auto rnd = [&](int lo, int hi) { return lo + (int)(gen() % (unsigned)(hi - lo + 1)); };
    for (int it = 0; it < 400; it++) {
        const int nx = it % 3 == 0 ? rnd(1, 60) : it % 3 == 1 ? rnd(60, 600) : rnd(600, 9000);
        const int ny = it % 2 ? rnd(1, 40) : rnd(40, 300), nchunk = (nx + 3) / 4, bucket = (nx + 63) / 64;
        MarchUnits u;
        u.K = 2 * rnd(2, 4);
        u.H = 8;
        u.nstrips = (nchunk + 27) / 28;
        u.nseg = std::max(1, std::min(rnd(1, 40), ny / 2));
        if (rnd(0, 2) == 0) {
            u.nl = std::min(rnd(0, 2), u.nstrips);
            u.nr = std::min(rnd(0, 2), u.nstrips - u.nl);
            u.nsegx = std::max(1, std::min(3 * u.nseg, ny / 2));
            const int he = ny >= 3 ? rnd(1, ny / 3) : 0;
            if (u.nseg >= 4 && he && 2 * he + (u.nseg - 2) * 2 <= ny) u.he = he;
        }
        std::vector<MarchEvent> ev;
        const bool low = rnd(0, 1);
        for (int k = rnd(1, 400); k > 0; k--)
            ev.push_back({low ? rnd(0, std::min(ny - 1, 5)) : rnd(0, ny - 1),
                          rnd(0, 1) ? rnd(0, nx - 1) : rnd(0, std::min(nx - 1, 130)), rnd(0, it % 5) == 0});
        const std::vector<MarchEvent> all = ev;
        const MarchEventCost c = march_event_cost(u, nx, ny, bucket, ev);
        double worst = 0.;
        int most = 0;
        for (int s = 0; s < u.nstrips; s++) {
            const int xs = 4 * march_cut(s, u.nstrips, nchunk);
            const int xe = s == u.nstrips - 1 ? nx : 4 * march_cut(s + 1, u.nstrips, nchunk);
            auto col = [&](int j) { return ((xs - u.H + j) % nx + nx) % nx; };
            unsigned long long cols = 0;
            for (int j = 0; j < 128; j++) cols |= 1ull << (col(j) / bucket);
            for (int k = 0; k < u.segs(s); k++) {
                const int y0 = u.row0(s, k, ny), y1 = u.row0(s, k + 1, ny);
                int rec = 0;
                bool twice = false;
                double v = 0.;
                for (int y = y0 - (u.K - 1); y < y1 + u.K - 1; y++) {
                    const int row = ((y % ny) + ny) % ny;
                    bool any = false;
                    double w = 0.;
                    int n = 0;
                    for (size_t i = 0; i < all.size(); i++) {
                        const MarchEvent &e = all[i];
                        if (e.row != row) continue;
                        n++;
                        w += e.source ? 2.5 : 1.;
                        any = any || (cols >> (e.x / bucket) & 1);
                        if (!e.source) {
                            rec += y >= y0 && y < y1 && e.x >= xs && e.x < xe;
                            continue;
                        }
                        int copies = 0;
                        for (int j = 0; j < 128; j++) copies += col(j) == e.x;
                        rec += copies;
                        for (size_t q = 0; q < i && copies; q++)
                            twice = twice || (all[q].source && all[q].row == row && all[q].x == e.x);
                    }
                    most = std::max(most, n);
                    if (any) v += w;
                }
                if (rec > MARCH_RECORDS || twice) worst = std::max(worst, v);
            }
        }
        if (worst != c.visits || most != c.row) return 1;
    }
    return 0;
}
"""


def test_event_cost_counts_every_unit(tmp_path):
    src = tmp_path / "h.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "h")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def _run(lbem, p, calls, steps_per_pass, storage="f32"):
    import torch

    s = lbem.Solver(p.shape, storage=storage)
    s.set_problem(p)
    lbem.lbem_set_temporal_blocking(s.h, steps_per_pass, -1)
    for n in calls:
        s.step(n)
    E, B = s.fields()
    tr = s.traces(p.rec_site.size)
    torch.cuda.synchronize()
    lbem.lbem_check_guards(s.h)
    s.close()
    return E.cpu().numpy(), B.cpu().numpy(), tr.cpu().numpy()


# a line of receivers puts more than 32 of them into each unit of its row; two sources share a site, others lie at the
# edges of the strips of 87 columns
@pytest.mark.gpu
@pytest.mark.parametrize("shape", [(40, 260), (23, 261)])
@pytest.mark.parametrize("medium", ["iso", "mu", "aniso", "pole", "walls", "walls_mu"])
def test_crowded_units_are_bitwise_identical_to_single_steps(lbem, shape, medium):
    eps, mu = W.random_medium(shape, 41, 1.2 if not medium.endswith("mu") else 1.0, mu=medium.endswith("mu"))
    p = W.Problem("crowd", 2, shape, eps, mu, 29)
    p.E0, p.B0 = W.random_fields(shape, 42, 0.3)
    ny, nx = shape
    rng = np.random.default_rng(43)
    if medium == "aniso":
        p.aniso = (2.0, 1.0)
    if medium == "pole":
        p.wp2 = rng.uniform(0.0, 0.5, shape)
        p.wr2 = rng.uniform(0.0, 0.1, shape)
        p.gamma = rng.uniform(0.0, 0.2, shape)
    if medium.startswith("walls"):
        p.bc, p.layer, p.gamma_max = (lbem.BC_PEC, lbem.BC_PMC, 0), 5, 0.3
    y = ny // 2
    p.src_site = np.array([y * nx + 50, y * nx + 50, 0, nx - 1, (y + 1) * nx + 87, (ny - 1) * nx + 174], np.int64)
    p.src_comp = np.full(p.src_site.size, 2, np.int32)
    p.src_amp = rng.standard_normal((p.src_site.size, 29))
    p.rec_site = np.concatenate([y * nx + np.arange(0, nx, 2), [0, nx - 1, (ny - 1) * nx]]).astype(np.int64)
    p.rec_comp = np.resize(np.array([2, 3, 4], np.int32), p.rec_site.size)
    ref = _run(lbem, p, [29], 1)
    for calls in ([29], [3, 5, 6, 8, 7]):
        for a, b in zip(_run(lbem, p, calls, 2), ref):
            np.testing.assert_array_equal(a, b, err_msg=f"{medium} {shape}, calls {calls}")


# The time of a call by default against launches of two steps (tile shape 0): a block of receivers took 6 to 16 times as
# long when it marched; taken by the same kernels, two runs differ by a few per cent.
@pytest.mark.gpu
@pytest.mark.parametrize("shape,block,storage", [((1024, 1024), 32, "f32"), ((1024, 1024), 32, "f16"), ((256, 256), 128, "f32")])
def test_crowded_grids_are_not_slower_than_launches_of_two_steps(lbem, shape, block, storage):
    import torch

    ny, nx = shape
    site = ((np.arange(block)[:, None] + ny // 3) * nx + np.arange(block)[None] + nx // 3).ravel().astype(np.int64)
    us = {}
    for tile in (0, -1):
        s = lbem.Solver(shape, storage=storage)
        lbem.lbem_set_medium(s.h, torch.full((nx * ny,), 2.0, device="cuda"))
        lbem.lbem_set_sources(s.h, [nx], [2], np.ones((1, 32), np.float32))
        lbem.lbem_set_receivers(s.h, site, np.full(site.size, 2, np.int32), 32)
        lbem.lbem_set_temporal_blocking(s.h, 2, tile)
        us[tile] = 1e30
        for _ in range(6):
            lbem.lbem_set_fields(s.h)
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            s.step(32)
            e[1].record()
            torch.cuda.synchronize()
            us[tile] = min(us[tile], e[0].elapsed_time(e[1]) * 1e3)
        s.close()
    assert us[-1] <= 1.2 * us[0], us
