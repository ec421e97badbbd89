"""FP32 Tersoff site terms, whose branches are taken by whole warps: atoms with
none to four list entries in registers next to atoms with more (records), in
ragged tiles, with bonds in the cutoff's edge and far from it, in single points
against the oracle at the stored FP32 configuration with the mixed path's
tolerance (1e-4, or 1e-6 of the largest force)."""
import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import f32_structure

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
