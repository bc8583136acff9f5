"""Kernel attributes are set once per CUDA device: the record behind every launcher (csrc/per_device.cuh, host code) keeps
one value per device, from any thread, and no launcher sets an attribute past it.  Two devices are played by numbers."""
import os
import re
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1108_2651_gb300", "csrc")

HARNESS = r"""
#include "per_device.cuh"
#include <cstdio>
#include <thread>
#include <vector>
int main() {
    struct Fit { int per_sm = 0, nsm = 0; };
    static lbk::PerDevice<Fit> at;
    int made[3] = {0, 0, 0};
    auto ask = [&](int dev, int fail, Fit *f) {
        return at.get(dev, [&](Fit &v) { made[dev]++; v.per_sm = 8; v.nsm = 100 + dev; return fail; }, f);
    };
    Fit f;
    if (ask(2, 7, &f) != 7 || made[2] != 1) return 1;          // a failure is reported and not kept
    if (ask(2, 0, &f) != 0 || made[2] != 2 || f.nsm != 102) return 2;
    int bad[64] = {};
    std::vector<std::thread> th;
    for (int k = 0; k < 64; k++)
        th.emplace_back([&, k] {
            Fit g;
            if (ask(k & 1, 0, &g) != 0 || g.per_sm != 8 || g.nsm != 100 + (k & 1)) bad[k] = 1;
        });
    for (auto &t : th) t.join();
    for (int b : bad) if (b) return 3;
    if (made[0] != 1 || made[1] != 1) return 4;                // each device's own, once
    if (at.get(1000, [](Fit &v) { v.nsm = 5; return 0; }, &f) != 0 || f.nsm != 5) return 5;
    return 0;
}
"""


def test_one_value_per_device(tmp_path):
    src = tmp_path / "h.cpp"
    src.write_text(HARNESS)
    exe = str(tmp_path / "h")
    subprocess.run(["g++", "-std=c++17", "-O1", "-pthread", "-I", CSRC, str(src), "-o", exe], check=True)
    assert subprocess.run([exe]).returncode == 0


def test_no_launcher_sets_attributes_for_the_process():
    """cudaFuncSetAttribute and the occupancy query appear in kernel_fit alone."""
    found = {}
    for f in sorted(os.listdir(CSRC)):
        n = len(re.findall(r"cudaFuncSetAttribute|cudaOccupancyMaxActiveBlocks", open(os.path.join(CSRC, f)).read()))
        if n:
            found[f] = n
    assert found == {"lbem_internal.cuh": 3}, found
