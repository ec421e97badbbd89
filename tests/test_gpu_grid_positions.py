"""Mixed many-body bands keep each atom's place in the cell as integers of a
grid with a remainder, and a neighbour's image as a lattice shift: cells
narrower than the list cutoff (shifts beyond +-1), atoms given outside the
cell by up to three lattice vectors (wraps inside and beyond the table of
shifts), sheared cells and a band that moves with kept lists, each against
the oracle at the stored FP32 configuration.  The tolerance is the mixed
path's own: max |dF| <= 1e-4 (or 1e-6 of the largest force)."""
import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import f32_structure, gpu_band

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_16721_gb300 as g
    g.build()
    return g


def _pot(g, oracle_mod, pot):
    if pot == "tersoff":
        return g.tersoff_potential(), oracle_mod.Tersoff()
    w = ci.nep_weights(seed=3)
    return g.nep_potential(w, 2.1), oracle_mod.NEP(w, rc=2.1)


def _carbon(kind, reps, shear, wraps, seed):
    Rg, hg, Rd, hd = ci.tersoff_endpoint_cells()
    R, h = ci.tile(Rg, hg, reps) if kind == "graphite" else ci.tile(Rd, hd, reps)
    rng = np.random.default_rng(seed)
    D = np.eye(3) + shear * np.array([[0.0, 1.0, -0.5], [0.0, 0.1, 1.0], [0.0, 0.0, 0.0]])
    R, h = R @ D, h @ D
    R = R + rng.normal(0.0, 0.04, R.shape)
    k = rng.integers(-wraps, wraps + 1, R.shape)
    return R + k @ h, h, k @ h


@pytest.mark.parametrize("wraps", [0, 1, 3])
@pytest.mark.parametrize("shear", [0.0, 0.3])
@pytest.mark.parametrize("reps", [(1, 1, 1), (2, 1, 3), (7, 5, 3)])
@pytest.mark.parametrize("kind", ["graphite", "diamond"])
@pytest.mark.parametrize("pot", ["tersoff", "nep"])
def test_single_points(g, oracle_mod, pot, kind, reps, shear, wraps):
    R, h, kh = _carbon(kind, reps, shear, wraps, 11)
    R, h = f32_structure(R, h)
    gp, op = _pot(g, oracle_mod, pot)
    E, F, V = g.evaluate([(R, h)], gp, g.MIXED)
    # the same periodic structure with its atoms inside the cell (the oracle's
    # NEP neighbour search takes nearest cells only)
    e, Fo, _ = op.evaluate(R - kh, h)
    assert np.max(np.abs(F[0] - Fo)) <= max(1e-4, 1e-6 * np.max(np.abs(Fo)))
    assert abs(E[0] - np.sum(e)) <= 1e-10 * np.sum(np.abs(e))


@pytest.mark.parametrize("reps", [(75, 1, 2), (90, 1, 2), (170, 1, 1), (2, 200, 1)])
def test_long_cells(g, oracle_mod, reps):
    """Extents on both sides of 205 A, where the grid becomes coarser, and of 410 and
    820 A."""
    R, h, kh = _carbon("diamond", reps, 0.0, 1, 11)
    R, h = f32_structure(R, h)
    e, Fo, _ = oracle_mod.Tersoff().evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], g.tersoff_potential(), g.MIXED)
    assert np.max(np.abs(F[0] - Fo)) <= max(1e-4, 1e-6 * np.max(np.abs(Fo)))
    assert abs(E[0] - np.sum(e)) <= 1e-10 * np.sum(np.abs(e))


@pytest.mark.parametrize("wraps", [1, 3])
@pytest.mark.parametrize("reps", [(2, 1, 1), (6, 4, 3)])
def test_moving_band(g, oracle_mod, reps, wraps):
    R0, h0, R1, h1 = ci.graphite_hexdiamond_path(reps)
    k = np.random.default_rng(5).integers(-wraps, wraps + 1, R0.shape)
    R0, R1 = R0 + k @ h0, R1 + k @ h1
    gb = gpu_band(g, R0, h0, R1, h1, 6, g.tersoff_potential(), k=0.1, dt=0.05, cell_filter=True,
                  precision=g.MIXED, noise=ci.interior_noise(4, 6, len(R0), 0.02))
    img = oracle_mod.AtomicImage(oracle_mod.Tersoff(), h0, len(R0), True)
    for steps in (1, 12):
        gb.step(steps)
        st = gb.get_state()
        E = gb.get_path()["energies"]
        gb.step(1)
        st2 = gb.get_state()
        for i in range(1, 5):
            Eo, Fo, _ = img(st["X"][i])
            s = np.max(np.abs(Fo))
            assert np.max(np.abs(st2["F"][i] - Fo)) <= max(1e-4, 1e-6 * s), (steps, i)
            assert abs(E[i] - Eo) <= 1e-10 * max(1.0, abs(Eo)), (steps, i)
