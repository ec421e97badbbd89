"""Band passes at the edges of a row tile (256 rows in FP64, 1024 in mixed
precision): bands whose n + 3 rows end just before, at and after one, two
steps against the oracle (FP64, 1e-9) and the FP64 path (mixed: FP32 rounding
of forces up to |F| moves a row by dt^2 F 2^-22 per step at most)."""
import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import gpu_band, oracle_band

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_16721_gb300 as g
    g.build()
    return g


def _ends(n, m):
    R, h = ci.fcc(ci.LJ_A, m, m, m)
    rng = np.random.default_rng(n)
    R0 = R[:n] + rng.normal(0.0, 0.02, (n, 3))
    return R0, h, R0 + rng.normal(0.0, 0.05, (n, 3)), ci.strained_cell(h, 3, 0.003)


@pytest.mark.parametrize("n", [252, 253, 254, 256, 257])
def test_fp64_row_tile_edges(g, oracle_mod, n):
    R0, h0, R1, h1 = _ends(n, 5)
    kw = dict(k=1.0, dt=0.005, cell_filter=True)
    gb = gpu_band(g, R0, h0, R1, h1, 4, g.lj_potential(), **kw)
    ob = oracle_band(oracle_mod, oracle_mod.LJ(), R0, h0, R1, h1, 4, **kw)
    gb.step(2)
    ob.step(2)
    st = gb.get_state()
    for i in (1, 2):
        s = max(1.0, np.max(np.abs(ob.F[i])))
        assert np.max(np.abs(st["F"][i] - ob.F[i])) <= 1e-9 * s
        assert np.max(np.abs(st["X"][i] - ob.X[i])) <= 1e-9 * np.max(np.abs(ob.X[i]))
        fn = ob.fneb[i - 1].reshape(st["Fneb"][i].shape)
        assert np.max(np.abs(st["Fneb"][i] - fn)) <= 1e-9 * s


@pytest.mark.parametrize("n", [1020, 1021, 1022, 1025])
def test_mixed_row_tile_edges(g, n):
    R0, h0, R1, h1 = _ends(n, 7)
    dt = 0.005
    kw = dict(k=1.0, dt=dt, cell_filter=True)
    bands = [gpu_band(g, R0, h0, R1, h1, 4, g.lj_potential(), precision=p, **kw)
             for p in (g.FP64, g.MIXED)]
    for b in bands:
        b.step(1)
    sd, sm = (b.get_state() for b in bands)
    F = np.max(np.abs(sd["Fneb"]))
    # the first move is dt^2 f_NEB: f_NEB carries the FP32 coordinates'
    # rounding times the pair stiffness (~1e3 eps/sigma^2, as in F) and F's own
    tol = dt * dt * (F * 2.0 ** -20 + 1e3 * 2.0 ** -23 * np.max(np.abs(sd["X"][:, :n]))) \
        + 4.0 * 2.0 ** -24 * np.max(np.abs(sd["X"][:, :n]))
    assert np.max(np.abs(sd["X"][1:3, :n] - sm["X"][1:3, :n])) <= tol
