"""The LJ cell walk (single points, the allocation-free call, bands without a
skin), which keeps screened candidates in shared memory and evaluates them a
warp at a time, with 1 to 32 lanes per atom by the band's size: sizes at the
edges of the lane rule and of a tile, an image beyond the 17-bit slot range
(two-word candidates), and a cell so dense that a thread's buffer fills within
a row.  FP64 against the oracle at the parity tests' 1e-10, FP32 at their
2e-6 of the largest force; totals beyond the oracle's reach against the
translation-invariant sum rules and the FP64 path."""
import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import f32_structure, perturbed

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_16721_gb300 as g
    g.build()
    return g


def _rel(a, b):
    return np.max(np.abs(np.asarray(a) - np.asarray(b))) / max(1.0, np.max(np.abs(b)))


@pytest.mark.parametrize("n", [1, 2, 3, 5, 33, 127, 129, 607, 609, 1215, 1217, 2431, 2433])
def test_lane_rule_edges(g, oracle_mod, n):
    m = max(1, int(np.ceil((n / 4.0) ** (1 / 3.0))))
    R, h = perturbed(*ci.fcc(ci.LJ_A, m, m, m), seed=n, amp=0.03, shear=0.02)
    R = R[:n]
    e, Fo, Vo = oracle_mod.LJ().evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], g.lj_potential(), g.FP64)
    assert abs(E[0] - e.sum()) <= 1e-10 * max(1.0, abs(e.sum()))
    assert _rel(F[0], Fo) <= 1e-10
    assert np.max(np.abs(V[0] - Vo)) <= 1e-10 * max(1.0, np.max(np.abs(Vo)))
    R32, h = f32_structure(R, h)
    e, Fo, Vo = oracle_mod.LJ().evaluate(R32, h)
    E, F, V = g.evaluate([(R32, h)], g.lj_potential(), g.MIXED)
    assert abs(E[0] - e.sum()) <= 1e-10 * max(1.0, abs(e.sum()))
    assert np.max(np.abs(F[0] - Fo)) <= max(1e-4, 2e-6 * np.max(np.abs(Fo)))


@pytest.mark.parametrize("precision", [0, 1])
def test_dense_cell_fills_the_buffer(g, oracle_mod, precision):
    """A crystal at a third of the LJ spacing under a long cutoff: ~1700
    neighbours per atom, hundreds of candidates in one stencil row."""
    R, h = perturbed(*ci.fcc(ci.LJ_A / 3.0, 6, 5, 7), seed=2, amp=0.005, shear=0.01)
    R, h = f32_structure(R, h)
    pot, op = g.lj_potential(1.0, 0.3, 2.0), oracle_mod.LJ(1.0, 0.3, 2.0)
    e, Fo, Vo = op.evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], pot, precision)
    assert abs(E[0] - e.sum()) <= 1e-10 * abs(e.sum())
    tol = 1e-10 * max(1.0, np.max(np.abs(Fo))) if precision == 0 else max(
        1e-4, 2e-6 * np.max(np.abs(Fo)))
    assert np.max(np.abs(F[0] - Fo)) <= tol


def test_two_word_candidates(g, oracle_mod):
    """137,180 atoms (above 2^17): sampled FP64 and mixed forces against the
    oracle, total force zero, the same reported energy on both paths."""
    R, h = perturbed(*ci.fcc(ci.LJ_A, 35, 35, 28), seed=6, amp=0.03)
    R, h = f32_structure(R, h)
    idx = np.random.default_rng(1).choice(len(R), 48, replace=False)
    Fo = oracle_mod.LJ().forces_sampled(R, h, idx)
    E, F, _ = g.evaluate([(R, h)], g.lj_potential(), g.FP64)
    assert _rel(F[0][idx], Fo) <= 1e-10
    assert np.all(np.abs(F[0].sum(0)) <= 1e-9 * len(R))
    Em, Fm, _ = g.evaluate([(R, h)], g.lj_potential(), g.MIXED)
    assert np.max(np.abs(Fm[0][idx] - Fo)) <= max(1e-4, 2e-6 * np.max(np.abs(Fo)))
    assert abs(E[0] - Em[0]) <= 1e-10 * abs(E[0])
