"""Block-int16 and 16-bit float states with NaN, infinite and huge values: the marched state, rounded in registers after
every second step, is the one that launches of two steps store, bit for bit."""
import numpy as np
import pytest

from paper_1108_2651_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _run(lbem, p, calls, tile, storage):
    import torch

    s = lbem.Solver(p.shape, storage=storage)
    s.set_problem(p)
    lbem.lbem_set_temporal_blocking(s.h, 2, tile)
    for n in calls:
        s.step(n)
    E, B = s.fields()
    tr = s.traces(p.rec_site.size)
    torch.cuda.synchronize()
    lbem.lbem_check_guards(s.h)
    s.close()
    return E.cpu().numpy(), B.cpu().numpy(), tr.cpu().numpy()


@pytest.mark.parametrize("storage", ["f16", "bf16", "i16b"])
def test_16bit_blocks_of_nan_and_huge_values(lbem, storage):
    shape = (33, 260)
    p = W.Problem("huge", 2, shape, W.random_medium(shape, 51, 1.2)[0], None, 24)
    p.E0, p.B0 = W.random_fields(shape, 52, 0.3)
    # (1e31 and 3e33 lie beyond block-int16's largest block, 1e-33 below its smallest)
    for k, v in enumerate([1e31, -3e33, np.inf, np.nan, 1e-33, 1e30]):
        p.E0[5 * k + 1, 40 * k + 7, 2] = v
    p.rec_site = np.random.default_rng(53).integers(0, 33 * 260, 12).astype(np.int64)
    p.rec_comp = np.resize(np.array([2, 3, 4], np.int32), 12)
    for calls in ([8], [24], [6, 10, 8]):
        ref = _run(lbem, p, calls, 0, storage)
        for a, b in zip(_run(lbem, p, calls, -1, storage), ref):
            np.testing.assert_array_equal(a, b, err_msg=f"{storage}, calls {calls}")
