"""Lennard-Jones in the caller's units: the same structure in reduced units and
with sigma = 2^-33 (1.2e-10, as in metres) and epsilon = 2^-69 gives the same
results, scaled.  Powers of two scale exactly, so the two differ by what the
bounds below allow for sums in another order at most (FP64 2^-40, FP32 2^-18 of
the largest value)."""
import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import gpu_band, lj_structures

pytestmark = pytest.mark.gpu

SIG, EPS = 2.0 ** -33, 2.0 ** -69


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_16721_gb300 as g
    g.build()
    return g


def _close(a, b, tol):
    assert np.max(np.abs(a - b)) <= tol * np.max(np.abs(b))


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("name", ["vacancy31", "one_cell", "triclinic240", "fcc2916"])
def test_points(g, name, precision):
    R, h = lj_structures()[name]
    tol = 2.0 ** -18 if precision else 2.0 ** -40
    E, F, V = g.evaluate([(R, h)], g.lj_potential(), precision)
    e, f, v = g.evaluate([(SIG * R, SIG * h)], g.lj_potential(EPS, SIG, 2.5 * SIG), precision)
    _close(e / EPS, E, 2.0 ** -40)
    _close(f[0] * SIG / EPS, F[0], tol)
    _close(v / EPS, V, tol)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("skin", [0.0, 0.3])
def test_bands(g, skin, precision):
    """End images as created and the energies of all; mixed bands after a move too
    (an FP64 move takes an FP32 seed of sums of squared forces: out of range here)."""
    R0, h0, R1, h1 = ci.lj_vacancy_hop(reps=(6, 6, 6))
    tol = 2.0 ** -18 if precision else 2.0 ** -40
    out = []
    for s, e in ((1.0, 1.0), (SIG, EPS)):
        band = gpu_band(g, s * R0, s * h0, s * R1, s * h1, 5, g.lj_potential(e, s, 2.5 * s),
                        k=e / s ** 2, dt=0.01 * s / e ** 0.5, maxstep=0.2 * s, cell_filter=False,
                        precision=precision, skin=skin * s)
        if precision:
            band.step(1)
        st = band.get_state()
        out.append((band.image_scalars()["E"] / e, st["F"][:, :-3] * s / e,
                    band.get_path()["energies"] / e))
        band.destroy()
    (E, F, P), (e, f, p) = out
    _close(e, E, tol)
    _close(f, F, tol)
    _close(p, P, tol)  # after a move by the forces
