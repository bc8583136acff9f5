"""lbem_autotune leaves several steps per launch on unless it timed them and they lost: a trial too short for a marching
launch, or a medium that the marching kernel does not take, does not switch it off.  Judged by the time of a call: on these
grids launches of one or two steps take at least 1.4 times as long as marching (1024^2: 6 against 2.3 us a step, 128^3: 62
against 40), so 1.2 times a fresh handle's time tells them apart."""
import numpy as np
import pytest

from paper_1108_2651_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _us(lbem, s, n):
    import torch

    best = 1e30
    for _ in range(6):
        e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        torch.cuda.synchronize()
        e[0].record()
        lbem.lbem_step(s.h, n)
        e[1].record()
        torch.cuda.synchronize()
        best = min(best, e[0].elapsed_time(e[1]) * 1e3)
    return best


def _solver(lbem, shape, mu=False):
    import torch

    s = lbem.Solver(shape)
    eps, mu_r = W.random_medium(shape, 11, 1.5, mu=mu)
    dev = lambda a: None if a is None else torch.as_tensor(np.asarray(a, np.float32).ravel(), device="cuda")
    lbem.lbem_set_medium(s.h, dev(eps), dev(mu_r))
    lbem.lbem_set_fields(s.h)
    return s


@pytest.mark.parametrize("shape", [(1024, 1024), (128, 128, 128)])
@pytest.mark.parametrize("trial", [1, 2, 4])
def test_short_trials_do_not_switch_marching_off(lbem, shape, trial):
    fresh, tuned = _solver(lbem, shape), _solver(lbem, shape)
    lbem.lbem_autotune(tuned.h, trial)
    a, b = _us(lbem, fresh, 48), _us(lbem, tuned, 48)
    assert b <= 1.2 * a, (a, b)
    fresh.close()
    tuned.close()


def test_a_medium_without_marching_does_not_switch_it_off(lbem):
    import torch

    shape = (128, 128, 128)
    fresh, tuned = _solver(lbem, shape), _solver(lbem, shape, mu=True)
    lbem.lbem_autotune(tuned.h, 6)
    eps = W.random_medium(shape, 11, 1.5)[0]
    lbem.lbem_set_medium(tuned.h, torch.as_tensor(np.asarray(eps, np.float32).ravel(), device="cuda"), None)
    a, b = _us(lbem, fresh, 48), _us(lbem, tuned, 48)
    assert b <= 1.2 * a, (a, b)
    fresh.close()
    tuned.close()
