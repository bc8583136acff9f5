"""A dispersive handle at the limit of device memory: without room for the second J plane it steps by launches of one and
two steps, J in place, to the same bits; without room for the others lbem_set_dispersion fails, holds nothing and works
once there is room."""
import ctypes
import os

import numpy as np
import pytest

from paper_1108_2651_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHAPE = (2048, 2048)
PLANE = 18 << 20  # a plane of 16 MB with its guard bands, in the allocator's 2 MB


def _cudart():
    home = os.environ.get("CUDA_HOME", "/usr/local/cuda")
    for name in (os.path.join(home, "lib64", "libcudart.so"), "libcudart.so"):
        try:
            rt = ctypes.CDLL(name)
            break
        except OSError:
            continue
    else:
        pytest.skip("no libcudart.so")
    rt.cudaMalloc.argtypes = [ctypes.POINTER(ctypes.c_void_p), ctypes.c_size_t]
    rt.cudaFree.argtypes = [ctypes.c_void_p]
    return rt


class _Leave:
    """Holds all free device memory but `left` bytes."""

    def __init__(self, rt, left):
        import torch

        self.rt, self.p = rt, ctypes.c_void_p()
        torch.cuda.synchronize()
        size = (torch.cuda.mem_get_info()[0] - left) >> 21 << 21
        if rt.cudaMalloc(ctypes.byref(self.p), size) != 0:
            pytest.skip("the free memory cannot be held in one piece")

    def __enter__(self):
        return self

    def __exit__(self, *a):
        self.rt.cudaFree(self.p)


def test_a_pole_without_room_for_a_second_plane(lbem):
    import torch

    rt = _cudart()
    n = SHAPE[0] * SHAPE[1]
    rng = np.random.default_rng(3)
    dev = lambda a: torch.as_tensor(np.asarray(a, np.float32).ravel(), device="cuda")
    eps = dev(W.random_medium(SHAPE, 4, 1.2)[0])
    pole = [dev(rng.uniform(0.0, hi, n)) for hi in (0.5, 0.1, 0.2)]
    E0 = dev(rng.standard_normal(3 * n))
    E, B = (torch.empty(3 * n, device="cuda") for _ in range(2))

    def solver():
        s = lbem.Solver(SHAPE)
        lbem.lbem_set_medium(s.h, eps)
        return s

    def run(s):
        lbem.lbem_set_fields(s.h, E0, None)
        for k in (8, 3, 2, 5, 1):
            s.step(k)
        lbem.lbem_fields(s.h, E, B)
        torch.cuda.synchronize()
        lbem.lbem_sync(s.h)
        lbem.lbem_check_guards(s.h)
        return E.clone(), B.clone()

    s = solver()
    lbem.lbem_set_dispersion(s.h, *pole)
    ref = run(s)
    lbem.lbem_set_temporal_blocking(s.h, 2, 0)  # (also loads the kernels that the next handle takes)
    for a, b in zip(run(s), ref):
        assert torch.equal(a, b)
    s.close()

    s = solver()
    with _Leave(rt, 9 * PLANE + PLANE // 2):
        lbem.lbem_set_dispersion(s.h, *pole)
        free = torch.cuda.mem_get_info()[0]
    assert free < PLANE  # there was no room for a tenth plane
    for a, b in zip(run(s), ref):
        assert torch.equal(a, b)
    s.close()

    s = solver()
    with _Leave(rt, 5 * PLANE + PLANE // 2):
        free = torch.cuda.mem_get_info()[0]
        with pytest.raises(lbem.LbemError):
            lbem.lbem_set_dispersion(s.h, *pole)
        assert torch.cuda.mem_get_info()[0] == free
        lbem.lbem_sync(s.h)
    lbem.lbem_set_dispersion(s.h, *pole)
    for a, b in zip(run(s), ref):
        assert torch.equal(a, b)
    s.close()
