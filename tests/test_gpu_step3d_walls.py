"""Single 3D steps with walls take little more than without: the walled kernel moves the same bytes, and its wall rule
touches the faces alone.  180 us a step at 192^3 without walls, 187 with; spilling registers it took 202."""
import pytest

pytestmark = pytest.mark.gpu


def test_walled_single_steps_cost_little_more(lbem):
    import torch

    shape = (192, 192, 192)
    us = {}
    for walls in (False, True):
        s = lbem.Solver(shape)
        lbem.lbem_set_medium(s.h, torch.full((192 ** 3,), 2.0, device="cuda"))
        if walls:
            lbem.lbem_set_boundaries(s.h, (1, 1, 1), 4, 0.2)
        lbem.lbem_set_fields(s.h)
        lbem.lbem_set_temporal_blocking(s.h, 1, -1)
        us[walls] = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            s.step(20)
            e[1].record()
            torch.cuda.synchronize()
            us[walls] = min(us[walls], e[0].elapsed_time(e[1]) * 50.0)
        s.close()
    assert us[True] <= 1.08 * us[False], us
