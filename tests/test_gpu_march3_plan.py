"""The 3D marching kernel's plan: the few numbers of segments that the host looks at hold the best of all, and a call does
not wait for the host to find it."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1108_2651_gb300", "csrc")

HARNESS = r"""
#include "march3_units.cuh"
#include <random>
using namespace lbk;
int main() {
    std::mt19937 gen(1);
    auto rnd = [&](int hi) { return 1 + (int)(gen() % (unsigned)hi); };
    const int K = 3, TY = 20;
    for (int i = 0; i < 20000; i++) {
        const int nx = rnd(i % 4 == 0 ? 40 : 700), ny = rnd(i % 4 == 2 ? 40 : 600), nz = rnd(i % 97 == 0 ? 20000 : 700);
        const int wave = i % 3 == 0 ? 152 : rnd(400);
        const March3Plan p = march3_plan(nx, ny, nz, K, TY, wave);
        if ((p.ntx - 1) * 28 >= nx || p.ntx * 28 < nx || (p.nty - 1) * 16 >= ny || p.nty * 16 < ny) return 1;
        if ((nz + p.nseg - 1) / p.nseg + 2 * (K - 1) > M3_PLANES) return 2;
        long long best = -1;
        int seg = 0;
        for (int n = (nz - 1) / (M3_PLANES - 2 * K) + 1; n <= nz; n++) {
            const long long cost = ((long long)p.ntx * p.nty * n + wave - 1) / wave * ((nz + n - 1) / n + 2 * (K - 1));
            if (best < 0 || cost < best) best = cost, seg = n;
        }
        if (best != p.planes || seg != p.nseg) return 3;
    }
    return 0;
}
"""


def test_plan_is_the_best_of_all_segment_numbers(tmp_path):
    src = tmp_path / "h.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "h")
    subprocess.run(["g++", "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


# a grid of very many planes, on which the search took 450 us of host time a call; the step itself takes 95 us
@pytest.mark.gpu
def test_a_step_does_not_wait_for_the_plan(lbem):
    import torch

    us = {}
    for spp in (1, 2):
        s = lbem.Solver((131072, 1, 4))
        lbem.lbem_set_medium(s.h, torch.full((4 * 131072,), 2.0, device="cuda"))
        lbem.lbem_set_fields(s.h)
        lbem.lbem_set_temporal_blocking(s.h, spp, -1)
        us[spp] = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(20):
                s.step(1)
            e[1].record()
            torch.cuda.synchronize()
            us[spp] = min(us[spp], e[0].elapsed_time(e[1]) * 50.0)
        s.close()
    assert us[2] <= 1.2 * us[1], us
