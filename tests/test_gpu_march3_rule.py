"""Which 3D grids march: flat and small ones, whose single steps are faster, keep those, and narrow ones, whose rows are
mostly padding, march and give the bits of single steps."""
import numpy as np
import pytest

from paper_1108_2651_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _us(lbem, s, n, calls):
    import torch

    best = 1e30
    for _ in range(8):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        for _ in range(calls):
            lbem.lbem_step(s.h, n)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) * 1e3 / calls)
    return best


# 3 x 250 x 460 took 34.0 us for three steps by marching and 26.4 by single steps, 30 x 24 x 96 14.0 and 12.3
@pytest.mark.parametrize("shape", [(3, 250, 460), (30, 24, 96)])
def test_marching_is_not_taken_where_single_steps_are_faster(lbem, shape):
    import torch

    us = {}
    for spp in (1, 2):
        s = lbem.Solver(shape)
        lbem.lbem_set_medium(s.h, torch.full((int(np.prod(shape)),), 2.0, device="cuda"))
        lbem.lbem_set_fields(s.h)
        lbem.lbem_set_temporal_blocking(s.h, spp, -1)
        us[spp] = _us(lbem, s, 30, 10)
        s.close()
    assert us[2] <= 1.07 * us[1], us


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(200, 40, 11), (300, 30, 5)])
def test_narrow_grids_are_bitwise_identical_to_single_steps(lbem, shape, walls):
    import torch

    p = W.Problem("narrow", 3, shape, W.random_medium(shape, 5, 1.0)[0], None, 14)
    p.E0, p.B0 = W.random_fields(shape, 6, 0.3)
    n = int(np.prod(shape))
    rng = np.random.default_rng(7)
    p.src_site = np.unique(np.concatenate([[0, shape[2] - 1, n - 1], rng.integers(0, n, 4)])).astype(np.int64)
    p.src_comp = rng.integers(0, 3, p.src_site.size).astype(np.int32)
    p.src_amp = rng.standard_normal((p.src_site.size, 14))
    p.rec_site = np.concatenate([p.src_site, rng.integers(0, n, 24)]).astype(np.int64)
    p.rec_comp = np.resize(np.arange(6, dtype=np.int32), p.rec_site.size)
    if walls:
        p.bc, p.layer, p.gamma_max = (1, 2, 1), 2, 0.2
    out = []
    for spp in (1, 2):
        s = lbem.Solver(shape)
        s.set_problem(p)
        lbem.lbem_set_temporal_blocking(s.h, spp, -1)
        s.step(14)
        E, B = s.fields()
        tr = s.traces(p.rec_site.size)
        torch.cuda.synchronize()
        lbem.lbem_check_guards(s.h)
        out.append([a.cpu().numpy() for a in (E, B, tr)])
        s.close()
    for a, b in zip(*out):
        np.testing.assert_array_equal(a, b)
