"""Cell lists of bands of at most 28,672 atoms are sorted in one launch (a
cluster of blocks per image), of larger ones or with very many bins in five:
sizes around what the cluster's threads take in one turn (4,096 atoms), at the
rule's line and beyond, with default bins, with more than one scan chunk of
them (16,384) and with more than the one launch takes.  Sampled forces against
the brute-force oracle at the step's own configuration (1e-10, FP64), with
lists rebuilt at every evaluation or kept."""
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


@pytest.mark.parametrize("reps,stretch,bin_scale,one", [
    ((2, 2, 2), 1.0, 1.0, True), ((8, 8, 16), 1.0, 1.0, True), ((8, 8, 16), 1.4, 0.3, True),
    ((10, 10, 11), 1.0, 0.3, True), ((16, 16, 28), 1.0, 1.0, True),
    ((16, 16, 28), 1.0, 0.3, True), ((19, 19, 20), 1.0, 1.0, False),
    ((16, 16, 28), 1.7, 0.3, False)])
@pytest.mark.parametrize("skin", [0.0, None])
def test_sorted_cell_list(g, oracle_mod, reps, stretch, bin_scale, one, skin):
    R0, h0, R1, h1 = ci.lj_vacancy_hop(stretch * ci.LJ_A, reps)
    n = len(R0)
    gb = gpu_band(g, R0, h0, R1, h1, 4, g.lj_potential(), k=1.0, dt=0.01, cell_filter=False,
                  noise=ci.interior_noise(4, 4, n, 0.02), bin_scale=bin_scale, skin=skin)
    assert (gb.launches_per_step() <= 9) == one
    gb.step(2)
    X = gb.get_state()["X"]
    gb.step(1)
    F = gb.get_state()["F"]
    idx = np.random.default_rng(7).choice(n, min(n, 24), replace=False)
    for i in (1, 2):
        Fo = oracle_mod.LJ().forces_sampled(X[i][:n], h0, idx)
        err = np.max(np.abs(F[i][idx] - Fo))
        assert err <= 1e-10 * max(1.0, np.max(np.abs(Fo))), (i, err)


@pytest.mark.parametrize("skin", [0.0, None])
@pytest.mark.parametrize("bin_scale", [1.0, 0.3])
def test_sorted_order_is_the_same(g, bin_scale, skin):
    """Runs repeat bit for bit: the order within a bin follows the atom
    index, not the order in which atoms arrived."""
    R0, h0, R1, h1 = ci.lj_vacancy_hop(ci.LJ_A, (10, 10, 10))
    kw = dict(k=1.0, dt=0.01, cell_filter=True, noise=ci.interior_noise(4, 5, len(R0), 0.02),
              bin_scale=bin_scale, skin=skin, precision=g.MIXED)
    st = []
    for _ in range(2):
        gb = gpu_band(g, R0, h0, R1, h1, 5, g.lj_potential(), **kw)
        gb.step(12)
        st.append(gb.get_state())
    assert np.array_equal(st[0]["X"], st[1]["X"]) and np.array_equal(st[0]["F"], st[1]["F"])


def test_more_images_than_clusters_points(g):
    """9,000 structures: each cluster sorts several, in more than one round of 32."""
    pot = g.lj_potential()
    few = [(np.array([[0.1 * k, 0.0, 0.0], [1.05 + 0.11 * k, 0.2, 0.0], [2.0, 2.0 + 0.05 * k, 1.0]]),
            np.eye(3) * (4.0 + 0.3 * k)) for k in range(9)]
    want = [g.evaluate([s], pot, g.FP64) for s in few]
    E, F, V = g.evaluate(few * 1000, pot, g.FP64)
    assert np.array_equal(E, np.tile([w[0][0] for w in want], 1000))
    for k in range(0, 9000, 7):
        w = want[k % 9]
        assert np.array_equal(F[k], w[1][0]) and np.array_equal(V[k], w[2][0])


@pytest.mark.parametrize("precision", [0, 1])
def test_more_images_than_clusters_bands(g, precision):
    """60 bands of 5 moving images whose lists are rebuilt at different steps:
    bit for bit as alone."""
    R0, h0, R1, h1 = ci.lj_vacancy_hop(ci.LJ_A, (2, 2, 2))
    kw = dict(k=1.0, dt=0.01, cell_filter=False, precision=precision, skin=0.1)

    def make(k):
        return gpu_band(g, R0, h0, R1, h1, 7, g.lj_potential(),
                        noise=ci.interior_noise(k, 7, len(R0), 0.002 * (k % 20)), **kw)

    bt = g.Batch(precision)
    bands = [make(k) for k in range(60)]
    for b in bands:
        bt.add(b)
    bt.step(40)
    stats = set()
    for k in (0, 7, 19, 31, 32, 33, 58, 59):
        alone = make(k)
        alone.step(40)
        a, b = alone.get_state(), bands[k].get_state()
        assert all(np.array_equal(a[q], b[q]) for q in ("X", "F", "Fneb", "virials"))
        stats.add(alone.list_stats()[0] if not isinstance(alone.list_stats(), dict)
                  else alone.list_stats()["builds"])
        alone.destroy()
    assert len(stats) > 2  # rebuilds differ between the bands
    bt.destroy()
