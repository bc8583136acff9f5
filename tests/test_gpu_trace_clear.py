"""lbem_set_fields clears the receivers' traces in the time of a memset, however few sites the grid has: on 16^2 the init
kernel's two blocks took 128 us for 4096 traces of 1000 samples, 15 us by memset; on 256^2 7 us alongside."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_small_grids_clear_many_traces_as_fast_as_a_memset(lbem):
    import torch

    us = {}
    for n in (16, 256):
        s = lbem.Solver((n, n))
        lbem.lbem_set_medium(s.h, torch.full((n * n,), 2.0, device="cuda"))
        lbem.lbem_set_receivers(s.h, np.arange(4096) % (n * n), np.full(4096, 2, np.int32), 1000)
        us[n] = 1e30
        for _ in range(6):
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record()
            for _ in range(10):
                lbem.lbem_set_fields(s.h)
            e[1].record()
            torch.cuda.synchronize()
            us[n] = min(us[n], e[0].elapsed_time(e[1]) * 100.0)
        s.close()
    assert us[16] <= 4.0 * us[256], us
