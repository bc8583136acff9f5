"""The marching kernel on widths that are not whole groups of four columns, which are copied element by element and may
have a wall inside a partial group, in every medium, and the tile kernels of a pole and a tensor beside it: the same bits
as single steps."""
import numpy as np
import pytest

from paper_1108_2651_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _problem(lbem, shape, medium, nsteps):
    eps, mu = W.random_medium(shape, 51, 1.2 if not medium.endswith("mu") else 1.0, mu=medium.endswith("mu"))
    p = W.Problem("edges", 2, shape, eps, mu, nsteps)
    p.E0, p.B0 = W.random_fields(shape, 52, 0.3)
    ny, nx = shape
    n = ny * nx
    rng = np.random.default_rng(53)
    if medium.endswith("aniso"):
        p.aniso = (2.0, 1.0)
    if medium == "pole":
        p.wp2 = rng.uniform(0.0, 0.5, shape)
        p.wr2 = rng.uniform(0.0, 0.1, shape)
        p.gamma = rng.uniform(0.0, 0.2, shape)
    if medium.startswith("walls"):
        p.bc, p.layer, p.gamma_max = (lbem.BC_PEC, lbem.BC_PMC, 0), min(5, min(shape) // 2), 0.3
    edge = [0, nx - 1, (ny - 1) * nx, n - 1, (ny // 2) * nx + nx - 2]
    p.src_site = np.unique(edge).astype(np.int64)
    p.src_comp = np.full(p.src_site.size, 2, np.int32)
    p.src_amp = rng.standard_normal((p.src_site.size, nsteps))
    p.rec_site = np.concatenate([edge, rng.integers(0, n, 12)]).astype(np.int64)
    p.rec_comp = np.resize(np.array([2, 3, 4], np.int32), p.rec_site.size)
    return p


def _run(lbem, p, calls, steps_per_pass, tile=-1):
    import torch

    s = lbem.Solver(p.shape)
    s.set_problem(p)
    lbem.lbem_set_temporal_blocking(s.h, steps_per_pass, tile)
    for n in calls:
        s.step(n)
    E, B = s.fields()
    tr = s.traces(p.rec_site.size)
    torch.cuda.synchronize()
    lbem.lbem_sync(s.h)
    lbem.lbem_check_guards(s.h)
    s.close()
    return E.cpu().numpy(), B.cpu().numpy(), tr.cpu().numpy()


@pytest.mark.parametrize("shape", [(9, 113), (40, 225), (64, 451), (31, 6)])
@pytest.mark.parametrize("medium", ["mu", "aniso", "pole", "walls", "walls_mu", "walls_aniso"])
def test_ragged_widths_in_every_medium(lbem, shape, medium):
    p = _problem(lbem, shape, medium, 27)
    ref = _run(lbem, p, [27], 1)
    # the default (marching), a split call, and for a pole also the tile kernel of two steps
    runs = [([27], -1), ([6, 7, 14], -1)] + ([([27], 0)] if medium in ("pole", "aniso") else [])
    for calls, tile in runs:
        for a, b in zip(_run(lbem, p, calls, 2, tile), ref):
            np.testing.assert_array_equal(a, b, err_msg=f"{medium} {shape}, calls {calls}, tile {tile}")
