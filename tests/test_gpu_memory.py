"""Device memory that does not suffice: the call that asked for too much says
so, and neither it nor any later call suffers from the refused allocation."""
import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import gpu_band

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_16721_gb300 as g
    g.build()
    return g


def _dimer(r, box):
    """Two LJ atoms in a box with many bins: a small structure with a cell list of
    up to 2^26 bins (0.5 GB)."""
    return np.array([[5.0, 5.0, 5.0], [5.0 + r, 5.0, 5.0]]), np.eye(3) * box


def test_calls_after_a_refused_allocation(g):
    R0, h0, R1, h1 = ci.lj_vacancy_hop()
    with pytest.raises(g.CfnebError) as e:  # hundreds of GB of image slots
        gpu_band(g, R0, h0, R1, h1, 5, g.lj_potential(), k=1.0, dt=0.01, n_max=40000000)
    assert e.value.status == g.ERR_OUT_OF_MEMORY
    E, F, V = g.evaluate([(R0, h0)], g.lj_potential(), g.FP64)
    band = gpu_band(g, R0, h0, R1, h1, 5, g.lj_potential(), k=1.0, dt=0.01)
    band.step(2)
    assert abs(band.get_path()["energies"][0] - E[0]) <= 1e-12 * abs(E[0])
    band.destroy()


def test_points_that_fit_one_by_one(g):
    """Six structures of 0.54 GB each with 2 GB free: one after the other."""
    import torch
    S = [_dimer(1.05 + 0.05 * k, 460.0) for k in range(6)]
    want = [g.evaluate([s], g.lj_potential(), g.FP64) for s in S]
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - (2 << 30), dtype=torch.uint8, device="cuda")
    try:
        E, F, V = g.evaluate(S, g.lj_potential(), g.FP64)
    finally:
        del hold
        torch.cuda.empty_cache()
    for k, (e, f, v) in enumerate(want):
        assert E[k] == e[0]
        assert np.array_equal(F[k], f[0]) and np.array_equal(V[k], v[0])


def test_a_group_of_points_is_bounded(g):
    """40 structures with 0.54 GB of bins each: a group takes 4 GB of them and
    little else, as another thread sees it."""
    import threading

    import torch
    S = [_dimer(1.05 + 0.01 * k, 460.0) for k in range(40)]
    torch.cuda.empty_cache()
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    least, done = [before], threading.Event()

    def watch():
        while not done.is_set():
            least[0] = min(least[0], torch.cuda.mem_get_info()[0])

    w = threading.Thread(target=watch)
    w.start()
    try:
        g.evaluate(S, g.lj_potential(), g.FP64)
    finally:
        done.set()
        w.join()
    assert before - least[0] <= 5 << 30
