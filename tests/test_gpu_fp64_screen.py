"""List builds of FP64 bands, which screen candidates on offsets rounded to
FP32 (with a margin that follows the bin size) and leave the FP64 test to the
force kernels: with fine, default and very coarse bins (offsets of many
cutoffs from a bin's centre, where the rounding is largest), rebuilt at every
evaluation or kept with a skin, the band follows the FP64 oracle at the
band-state tolerance of the parity tests."""
import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import gpu_band, lj_band_case, oracle_band

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


@pytest.mark.parametrize("skin", [0.0, None])
@pytest.mark.parametrize("bin_scale", [0.3, 1.0, 8.0])
@pytest.mark.parametrize("pot", ["lj", "tersoff"])
def test_fp64_lists_screened_in_fp32(g, oracle_mod, pot, bin_scale, skin):
    if pot == "lj":
        R0, h0, R1, h1 = lj_band_case(strain_seed=3)
        kw = dict(k=1.0, dt=0.01, cell_filter=True)
        gp, op, N = g.lj_potential(), oracle_mod.LJ(), 5
    else:
        R0, h0, R1, h1 = ci.graphite_hexdiamond_path((4, 3, 2))
        kw = dict(k=0.1, dt=0.05, cell_filter=True,
                  noise=ci.interior_noise(3, 5, len(R0), 0.02))
        gp, op, N = g.tersoff_potential(), oracle_mod.Tersoff(), 5
    gb = gpu_band(g, R0, h0, R1, h1, N, gp, bin_scale=bin_scale, skin=skin, **kw)
    ob = oracle_band(oracle_mod, op, R0, h0, R1, h1, N, **kw)
    gb.step(4)
    ob.step(4)
    st = gb.get_state()
    for i in range(1, N - 1):
        assert _rel(st["F"][i], ob.F[i]) <= 1e-9, i
        assert _rel(st["X"][i], ob.X[i]) <= 1e-9, i


@pytest.mark.parametrize("reps", [(2, 2, 2), (3, 4, 5), (6, 6, 7), (11, 9, 10)])
def test_fp64_lj_lists_with_lanes(g, oracle_mod, reps):
    """FP64 LJ bands with neighbour lists give an atom 32 to 4 lanes by their
    size (31, 239, 1007 and 3959 atoms, each with a ragged last tile): one
    step from displaced positions against the oracle."""
    R0, h0, R1, h1 = ci.lj_vacancy_hop(ci.LJ_A, reps)
    h1s = ci.strained_cell(h1, 3, 0.01)
    kw = dict(k=1.0, dt=0.01, cell_filter=True, noise=ci.interior_noise(4, 4, len(R0), 0.02))
    gb = gpu_band(g, R0, h0, ci.affine(R1, h1, h1s), h1s, 4, g.lj_potential(), **kw)
    ob = oracle_band(oracle_mod, oracle_mod.LJ(), R0, h0, ci.affine(R1, h1, h1s), h1s, 4, **kw)
    gb.step(1)
    ob.step(1)
    st = gb.get_state()
    for i in (1, 2):
        assert _rel(st["F"][i], ob.F[i]) <= 1e-10, i
        assert _rel(st["virials"][i], ob.info[i]["V"]) <= 1e-10, i
