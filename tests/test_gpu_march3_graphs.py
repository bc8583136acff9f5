"""3D steps replayed from CUDA graphs: marching is not taken where the graph's single steps are faster, which they are on
more grids than in a stream (64^3 7.5 us a step in a graph, 8.2 in a stream; marching 8.6 and 7.9)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(32, 32, 32), (64, 64, 64)])
def test_graphs_are_not_slower_than_graphs_of_single_steps(lbem, shape):
    import torch

    n = int(np.prod(shape))
    us, st = {1: 1e30, 2: 1e30}, torch.cuda.Stream()
    solvers = {}
    for spp in us:
        s = solvers[spp] = lbem.Solver(shape, stream=st.cuda_stream)
        lbem.lbem_set_medium(s.h, torch.full((n,), 2.0, device="cuda"))
        lbem.lbem_set_fields(s.h)
        lbem.lbem_set_temporal_blocking(s.h, spp, -1)
        lbem.lbem_set_graphs(s.h, True)
    for _ in range(15):
        for spp, s in solvers.items():
            e = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
            torch.cuda.synchronize()
            e[0].record(st)
            s.step(300)
            e[1].record(st)
            torch.cuda.synchronize()
            us[spp] = min(us[spp], e[0].elapsed_time(e[1]) / 0.3)
    for s in solvers.values():
        s.close()
    assert us[2] <= 1.1 * us[1], us  # (32^3 by marching: 1.2 times as long)
