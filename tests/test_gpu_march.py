"""The marching kernel (8 steps per launch, the default for calls of at least 3 steps) against single steps.

Every site update is the single-step kernel's arithmetic in its order, so E, B and the receiver traces are
bit-identical for every grid, step count and split of the steps into calls.  The grids lie at the kernel's edges: strips
of up to 112 columns (4 * 28) with 8 columns of halo, rows whose last group of four is partial, segments of two rows,
grids smaller than a halo.
"""
import numpy as np
import pytest

from paper_1108_2651_gb300 import lbem, workloads as W

pytestmark = pytest.mark.gpu


def _problem(shape, seed, nsteps, mu=False):
    eps, mu_r = W.random_medium(shape, seed, 1.2 if not mu else 1.0, mu=mu)
    p = W.Problem("march", 2, shape, eps, mu_r, nsteps)
    p.E0, p.B0 = W.random_fields(shape, seed + 1, 0.3)
    ny, nx = shape
    n = ny * nx
    rng = np.random.default_rng(seed + 2)
    corners = [0, nx - 1, (ny - 1) * nx, n - 1, (ny // 2) * nx + min(nx - 1, 112)]
    p.src_site = np.unique(np.concatenate([corners, rng.integers(0, n, 3)])).astype(np.int64)
    p.src_comp = np.full(p.src_site.size, 2, np.int32)
    p.src_amp = rng.standard_normal((p.src_site.size, nsteps))
    p.rec_site = np.concatenate([corners, rng.integers(0, n, 20)]).astype(np.int64)  # two may share a site
    p.rec_comp = np.resize(np.array([2, 3, 4], np.int32), p.rec_site.size)
    return p


def _run(p, calls, steps_per_pass=None, graphs=False, storage="f32", shape=-1):
    import torch

    stream = torch.cuda.Stream() if graphs else None
    s = lbem.Solver(p.shape, storage=storage, stream=stream.cuda_stream if stream else None)
    s.set_problem(p)
    if steps_per_pass:
        lbem.lbem_set_temporal_blocking(s.h, steps_per_pass, shape)
    if graphs:
        lbem.lbem_set_graphs(s.h, True)
    for n in calls:
        s.step(n)
    E, B = s.fields()
    tr = s.traces(p.rec_site.size)
    torch.cuda.synchronize()
    lbem.lbem_sync(s.h)
    lbem.lbem_check_guards(s.h)
    s.close()
    return E.cpu().numpy(), B.cpu().numpy(), tr.cpu().numpy()


@pytest.mark.parametrize("shape", [(1, 1), (1, 300), (2, 3), (3, 112), (5, 113), (9, 116), (17, 224), (40, 225),
                                   (300, 5), (64, 451), (131, 1000), (700, 337)])
def test_march_is_bitwise_identical_to_single_steps(lbem, shape):
    p = _problem(shape, 700 + shape[1], 43)
    ref = _run(p, [43], steps_per_pass=1)
    for calls in ([43], [8, 35], [16, 16, 11], [3, 4, 5, 6, 7, 9, 9], [1, 2, 40]):
        for graphs in (False, True):
            got = _run(p, calls, graphs=graphs)
            for a, b in zip(got, ref):
                np.testing.assert_array_equal(a, b, err_msg=f"{shape}, calls {calls}, graphs {graphs}")


@pytest.mark.parametrize("shape", [(1, 4), (7, 116), (33, 260), (300, 452)])
@pytest.mark.parametrize("medium", ["mu", "aniso", "pole", "walls", "walls_mu", "walls_aniso"])
def test_march_media_are_bitwise_identical_to_single_steps(lbem, shape, medium):
    p = _problem(shape, 800 + shape[1], 29, mu=medium.endswith("mu"))
    rng = np.random.default_rng(5)
    if medium.endswith("aniso"):
        p.aniso = (2.0, 1.0)
    if medium == "pole":
        p.wp2 = rng.uniform(0.0, 0.5, shape)
        p.wr2 = rng.uniform(0.0, 0.1, shape)
        p.gamma = rng.uniform(0.0, 0.2, shape)
    if medium.startswith("walls"):
        p.bc, p.layer, p.gamma_max = (lbem.BC_PEC, lbem.BC_PMC, 0), min(5, min(shape) // 2), 0.3
    ref = _run(p, [29], steps_per_pass=1)
    for calls, graphs in (([29], False), ([6, 8, 15], True), ([3, 4, 5, 17], False)):
        for a, b in zip(_run(p, calls, graphs=graphs), ref):
            np.testing.assert_array_equal(a, b, err_msg=f"{medium} {shape}, calls {calls}")


@pytest.mark.parametrize("shape", [(1, 4), (7, 116), (33, 260), (300, 1028)])
@pytest.mark.parametrize("storage", ["f16", "bf16", "i16b"])
def test_march_16bit_equals_launches_of_two_steps(lbem, shape, storage):
    """(300, 1028): strips' edges long enough that a block exponent taken from a spoilt halo column shows.)"""
    p = _problem(shape, 900 + shape[1], 30)
    for calls in ([30], [8, 22], [4, 6, 10, 10], [3, 27]):
        ref = _run(p, calls, steps_per_pass=2, shape=0, storage=storage)
        for a, b in zip(_run(p, calls, storage=storage), ref):
            np.testing.assert_array_equal(a, b, err_msg=f"{storage} {shape}, calls {calls}")


# grids that the rule on sizes gives to the 3D kernel (28 x 16 columns a tile, segments of the planes): one tile, a tile
# that is a column or a row too wide, one plane a segment, an odd remainder of everything, several waves of blocks
@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("shape", [(220, 16, 28), (64, 64, 85), (90, 81, 84), (3, 250, 460), (75, 61, 90),
                                   (131, 119, 131)])
def test_march_3d_is_bitwise_identical_to_single_steps(lbem, shape, walls):
    nsteps = 14
    eps, _ = W.random_medium(shape, 5, 1.0)
    p = W.Problem("march3", 3, shape, eps, None, nsteps)
    p.E0, p.B0 = W.random_fields(shape, 6, 0.3)
    nz, ny, nx = shape
    n = nz * ny * nx
    rng = np.random.default_rng(7)
    corners = [0, nx - 1, (ny - 1) * nx, n - 1, min(nx - 1, 28), (nz // 2 * ny + min(ny - 1, 16)) * nx]
    p.src_site = np.unique(np.concatenate([corners, rng.integers(0, n, 4)])).astype(np.int64)
    p.src_comp = rng.integers(0, 3, p.src_site.size).astype(np.int32)
    p.src_amp = rng.standard_normal((p.src_site.size, nsteps))
    p.rec_site = np.concatenate([corners, rng.integers(0, n, 24)]).astype(np.int64)
    p.rec_comp = np.resize(np.arange(6, dtype=np.int32), p.rec_site.size)
    if walls:
        p.bc, p.layer, p.gamma_max = (1, 2, 1), min(3, min(shape) // 2), 0.2
    ref = _run(p, [nsteps], steps_per_pass=1)
    for calls in ([nsteps], [3, 4, 5, 2]):
        for graphs in (False, True):
            for a, b in zip(ref, _run(p, calls, graphs=graphs)):
                np.testing.assert_array_equal(a, b)


# the 3D adjoint: sigma of every step or of checkpointed segments, three steps per launch or one; the last shape is too
# small for three
@pytest.mark.parametrize("shape", [(90, 81, 84), (75, 61, 90), (9, 20, 37)])
def test_march_3d_adjoint_is_bitwise_identical_to_single_steps(lbem, shape):
    import torch

    from paper_1108_2651_gb300.autograd import receiver_traces

    n = int(np.prod(shape))
    eps0 = torch.from_numpy(W.random_medium(shape, 5, 1.0)[0].astype(np.float32)).cuda()

    def run(nsteps, every, steps_per_pass, repeat=1):
        rng = np.random.default_rng(8)
        p = W.Problem("march3", 3, shape, None, None, nsteps)
        p.src_site = np.unique(np.concatenate([[0, n - 1], rng.integers(0, n, 4)])).astype(np.int64)
        p.src_comp = np.resize(np.arange(3, dtype=np.int32), p.src_site.size)
        p.src_amp = rng.standard_normal((p.src_site.size, nsteps))
        p.rec_site = np.concatenate([p.src_site, rng.integers(0, n, 24)]).astype(np.int64)
        p.rec_comp = np.resize(np.arange(6, dtype=np.int32), p.rec_site.size)
        cot = torch.from_numpy(rng.standard_normal((p.rec_site.size, nsteps)).astype(np.float32)).cuda()
        s = lbem.Solver(shape)
        lbem.lbem_set_temporal_blocking(s.h, steps_per_pass, -1)
        for _ in range(repeat):  # a second run takes over the first one's buffers
            eps = eps0.clone().requires_grad_(True)
            tr = receiver_traces(eps, s, p, checkpoint_every=every)
            tr.backward(cot)
        torch.cuda.synchronize()
        lbem.lbem_check_guards(s.h)
        s.close()
        return tr.detach().cpu().numpy(), eps.grad.cpu().numpy()

    for nsteps, everys in ((14, (14, 4, 1)), (241, (241, 16))):  # 241 steps, a state kept every 16
        ref = run(nsteps, nsteps, 1)
        assert np.abs(ref[1]).max() > 0
        for every in everys:
            for spp, repeat in ((1, 1), (2, 2)):
                for a, b in zip(ref, run(nsteps, every, spp, repeat)):
                    np.testing.assert_array_equal(a, b)
