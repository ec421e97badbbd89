"""FP32 Tersoff site terms, whose branches are taken by whole warps: atoms with
none to four list entries in registers next to atoms with more (records), in
ragged tiles, with bonds in the cutoff's edge and far from it, in single points
against the oracle at the stored FP32 configuration with the mixed path's
tolerance (1e-4, or 1e-6 of the largest force)."""
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


def _carbon(kind, reps, drop, seed):
    Rg, hg, Rd, hd = ci.tersoff_endpoint_cells()
    R, h = ci.tile(Rg, hg, reps) if kind == "graphite" else ci.tile(Rd, hd, reps)
    rng = np.random.default_rng(seed)
    sigma = {"graphite": 0.03, "diamond": 0.03, "dense": 0.03, "disordered": 0.12, "edge": 0.05,
             "sparse": 0.05}[kind]
    scale = {"dense": 0.86, "edge": 1.27}.get(kind, 1.0)  # bonds of 1.96 A: inside R +- D
    R, h = scale * R, scale * h
    R = R + rng.normal(0.0, sigma, R.shape)
    keep = rng.permutation(len(R))[:len(R) - drop]
    if kind == "sparse":  # half of the atoms: zero to four neighbours
        keep = rng.permutation(len(R))[:len(R) // 2 - drop]
    return R[np.sort(keep)], h


@pytest.mark.parametrize("reps,drop", [((1, 1, 1), 0), ((2, 1, 2), 1), ((3, 2, 3), 15),
                                       ((4, 4, 4), 0), ((6, 5, 4), 3)])
@pytest.mark.parametrize("kind", ["graphite", "diamond", "dense", "disordered", "edge", "sparse"])
def test_points(g, oracle_mod, kind, reps, drop):
    if kind == "sparse" and len(range(8 * np.prod(reps) // 2 - drop)) < 2:
        drop = 0
    R, h = f32_structure(*_carbon(kind, reps, drop, 3))
    e, Fo, Vo = oracle_mod.Tersoff().evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], g.tersoff_potential(), g.MIXED)
    assert np.max(np.abs(F[0] - Fo)) <= max(1e-4, 1e-6 * np.max(np.abs(Fo)))
    assert abs(E[0] - e.sum()) <= 1e-10 * max(1.0, np.abs(e).sum())
    assert np.max(np.abs(V[0] - Vo)) <= 1e-4 * len(R)


def _sharp(g, oracle_mod):
    """Carbon's constants with a cutoff of no width (D = 0) at 2 A."""
    q = dict(oracle_mod.TERSOFF_C1988, R=2.0, D=0.0)
    order = ["A", "B", "lambda1", "lambda2", "beta", "n", "c", "d", "h", "R", "D"]
    return g.tersoff_potential([q[k] for k in order]), oracle_mod.Tersoff(q)


@pytest.mark.parametrize("kind,reps,drop", [("graphite", (2, 1, 2), 1), ("diamond", (3, 2, 3), 15),
                                            ("dense", (2, 2, 2), 0), ("sparse", (4, 4, 4), 0)])
def test_sharp_cutoff_points(g, oracle_mod, kind, reps, drop):
    """Entries that an atom does not have stay outside a cutoff of no width."""
    pot, o = _sharp(g, oracle_mod)
    R, h = f32_structure(*_carbon(kind, reps, drop, 3))
    e, Fo, Vo = o.evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], pot, g.MIXED)
    assert np.max(np.abs(F[0] - Fo)) <= max(1e-4, 1e-6 * np.max(np.abs(Fo)))
    assert np.max(np.abs(V[0] - Vo)) <= 1e-4 * len(R)


def test_sharp_cutoff_step_energies(g, oracle_mod):
    """The end images' step energies: 63 atoms leave half of a block without one.
    FP32 site energies: a few 1e-7 of each atom's energy and of a warp's sum."""
    pot, o = _sharp(g, oracle_mod)
    R0, h0, R1, h1 = ci.diamond_vacancy_hop(reps=(2, 2, 2))
    R0, R1 = f32_structure(R0, h0)[0], f32_structure(R1, h1)[0]
    band = gpu_band(g, R0, h0, R1, h1, 3, pot, k=0.1, dt=0.05, precision=g.MIXED)
    E = band.image_scalars()["E"]
    band.destroy()
    e0, e1 = o.evaluate(R0, h0)[0].sum(), o.evaluate(R1, h1)[0].sum()
    assert abs(E[0] - e0) <= 1e-6 * abs(e0)
    assert abs(E[2] - e1) <= 1e-6 * abs(e1)


@pytest.mark.parametrize("product", [4e37, 8.6e37, 1.2e38, 1.6e38])
def test_large_bond_order_argument(g, oracle_mod, product):
    """Three atoms in the cutoff's edge with (beta zeta)^n zeta about 2^126 to 2^127,
    where FP32 has no normal reciprocal: forces through db/dzeta."""
    n, zeta = 50.0, 0.5  # f_C = 1/2 at r = R, g = 1
    beta = (product / zeta) ** (1.0 / n) / zeta
    par = [1393.6, 346.74, 3.4879, 2.2119, beta, n, 0.0, 1.0, -0.57, 1.95, 0.15]
    R = 5.0 + 1.95 * np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [0.5, 0.75 ** 0.5, 0.0]])
    R, h = f32_structure(R, np.eye(3) * 12.0)
    names = ["A", "B", "lambda1", "lambda2", "beta", "n", "c", "d", "h", "R", "D"]
    e, Fo, Vo = oracle_mod.Tersoff(dict(zip(names, par))).evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], g.tersoff_potential(par), g.MIXED)
    assert np.max(np.abs(F[0] - Fo)) <= 1e-4
