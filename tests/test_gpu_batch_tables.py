"""A batch's work tables outlive a change of variant: the marching kernel's unit table (variant 16) stays the batch's own
when the strip kernels' table (14, 15) is made or grows after it, and is freed with the batch.  Variants taken in any
order, and the autotuner after a marching step, give each member the bits it gets when stepped alone."""
import numpy as np
import pytest

from paper_1108_2651_gb300 import workloads as W

pytestmark = pytest.mark.gpu


def _members(lbem, stream, nsteps):
    probs = [W.heterogeneous_2d(N, seed=70 + N, nsteps=nsteps, sigma=min(20.0, N / 8.0), nrec=4, rec_radius=N // 4)
             for N in (64, 99, 130, 257)]
    out = []
    for p in probs:
        s = lbem.Solver(p.shape, stream=stream)
        s.set_problem(p)
        out.append(s)
    return probs, out


def _read(s, p):
    import torch

    E, B = s.fields()
    tr = s.traces(p.rec_site.size)
    torch.cuda.synchronize()
    return E.cpu().numpy(), B.cpu().numpy(), tr.cpu().numpy()


# (variant, steps) in turn; "autotune" times every variant and keeps the fastest
@pytest.mark.parametrize("plan", [[(16, 9), (15, 8), (14, 6), (16, 12), (9, 3), (16, 8)],
                                  [(16, 9), "autotune", (16, 10), (15, 4), (16, 5)]])
def test_batch_variants_in_any_order(lbem, plan):
    import torch

    n = sum(q[1] for q in plan if q != "autotune")
    st = torch.cuda.Stream()
    probs, alone = _members(lbem, st.cuda_stream, n)
    ref = []
    for s, p in zip(alone, probs):
        lbem.lbem_set_temporal_blocking(s.h, 1, -1)
        s.step(n)
        ref.append(_read(s, p))
        s.close()
    _, ss = _members(lbem, st.cuda_stream, n)
    b = lbem.lbem_batch_create([s.h for s in ss], st.cuda_stream)
    for q in plan:
        if q == "autotune":
            lbem.lbem_batch_autotune(b, 4)
            for s, p in zip(ss, probs):  # (its trials record into the receivers' traces)
                assert lbem.lbem_time(s.h) == 9
        else:
            lbem.lbem_batch_set_variant(b, q[0])
            lbem.lbem_batch_step(b, q[1])
    for s, p, r in zip(ss, probs, ref):
        lbem.lbem_check_guards(s.h)
        for a, q in zip(_read(s, p), r):
            np.testing.assert_array_equal(a, q, err_msg=f"{plan}, {p.shape}")
    lbem.lbem_batch_destroy(b)
    for s in ss:
        s.close()


def test_batch_gives_its_tables_back(lbem):
    """Device memory in use does not grow with batches that marched and were destroyed."""
    import torch

    st = torch.cuda.Stream()
    _, ss = _members(lbem, st.cuda_stream, 400)
    free = []
    for k in range(260):  # (a leaked table of this batch takes 512 bytes to 2 MB of the driver's pool)
        b = lbem.lbem_batch_create([s.h for s in ss], st.cuda_stream)
        lbem.lbem_batch_set_variant(b, 16)
        lbem.lbem_batch_step(b, 1)
        lbem.lbem_batch_destroy(b)
        if k in (9, 259):
            torch.cuda.synchronize()
            free.append(torch.cuda.mem_get_info()[0])
    for s in ss:
        s.close()
    assert free[0] == free[1], free
