"""Neighbour lists built by several lanes per atom (FP64 bands whose tiles hold
fewer atoms than threads, and small mixed carbon bands): cells narrower than
the stencil, ragged last tiles, dense cells with many entries and sizes at the
line between the two forms, rebuilt at every evaluation or kept, against the
oracle at the step's own configuration (FP64 1e-10; mixed 1e-4 or 1e-6 of the
largest force), and an overflowing list reported as such."""
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


@pytest.mark.parametrize("skin", [0.0, None])
@pytest.mark.parametrize("reps,images,precision", [
    ((1, 1, 1), 4, "fp64"), ((3, 2, 1), 5, "fp64"), ((7, 5, 4), 4, "fp64"), ((1, 1, 1), 4, "mixed"),
    ((3, 2, 1), 5, "mixed"), ((7, 5, 4), 5, "mixed"), ((16, 11, 14), 3, "mixed")])
def test_carbon(g, oracle_mod, reps, images, precision, skin):
    R0, h0, R1, h1 = ci.graphite_hexdiamond_path(reps)
    n = len(R0)
    mixed = precision == "mixed"
    gb = gpu_band(g, R0, h0, R1, h1, images, g.tersoff_potential(), k=0.1, dt=0.02,
                  cell_filter=True, precision=g.MIXED if mixed else g.FP64, skin=skin,
                  noise=ci.interior_noise(3, images, n, 0.02))
    gb.step(2)
    X = gb.get_state()["X"]
    gb.step(1)
    F = gb.get_state()["F"]
    img = oracle_mod.AtomicImage(oracle_mod.Tersoff(), h0, n, True)
    for i in range(1, images - 1):
        _, Fo, _ = img(X[i])
        s = np.max(np.abs(Fo))
        tol = max(1e-4, 1e-6 * s) if mixed else 1e-10 * max(1.0, s)
        assert np.max(np.abs(F[i] - Fo)) <= tol, i


@pytest.mark.parametrize("reps", [(2, 2, 2), (3, 3, 2), (5, 5, 6), (9, 9, 10)])
def test_lj(g, oracle_mod, reps):
    R0, h0, R1, h1 = ci.lj_vacancy_hop(ci.LJ_A, reps)
    n = len(R0)
    gb = gpu_band(g, R0, h0, R1, h1, 5, g.lj_potential(), k=1.0, dt=0.01, cell_filter=False,
                  noise=ci.interior_noise(4, 5, n, 0.03))
    gb.step(2)
    X = gb.get_state()["X"]
    gb.step(1)
    F = gb.get_state()["F"]
    idx = np.random.default_rng(7).choice(n, min(n, 40), replace=False)
    for i in (1, 2, 3):
        Fo = oracle_mod.LJ().forces_sampled(X[i][:n], h0, idx)
        assert np.max(np.abs(F[i][idx] - Fo)) <= 1e-10 * max(1.0, np.max(np.abs(Fo))), i


@pytest.mark.parametrize("precision", ["fp64", "mixed"])
def test_overflow_is_reported(g, precision):
    """More than 16 list entries per atom: an error, not a truncated list."""
    Rg, hg, Rd, hd = ci.tersoff_endpoint_cells()
    R, h = ci.tile(Rd, hd, (3, 2, 2))
    R, h = 0.6 * R, 0.6 * h
    with pytest.raises(g.CfnebError) as e:
        gb = gpu_band(g, R, h, R + 0.01, h, 4, g.tersoff_potential(), k=0.1, dt=0.01,
                      cell_filter=True, precision=g.MIXED if precision == "mixed" else g.FP64)
        gb.step(1)
    assert e.value.status == g.ERR_NBR_OVERFLOW


@pytest.mark.parametrize("reps", [(2, 2, 2), (5, 5, 5), (8, 8, 9), (17, 17, 17)])
def test_lj_mixed(g, oracle_mod, reps):
    """Mixed LJ bands: sets of 3 to 462 tiles, split over 16 blocks to none."""
    R0, h0, R1, h1 = ci.lj_vacancy_hop(ci.LJ_A, reps)
    n = len(R0)
    gb = gpu_band(g, R0, h0, R1, h1, 5, g.lj_potential(), k=1.0, dt=0.01, cell_filter=False,
                  precision=g.MIXED, noise=ci.interior_noise(4, 5, n, 0.03))
    gb.step(2)
    X = gb.get_state()["X"]
    gb.step(1)
    F = gb.get_state()["F"]
    idx = np.random.default_rng(7).choice(n, min(n, 40), replace=False)
    for i in (1, 2, 3):
        Fo = oracle_mod.LJ().forces_sampled(X[i][:n], h0, idx)
        assert np.max(np.abs(F[i][idx] - Fo)) <= 1e-4, i
