"""Single points in groups (one allocation and one launch per kernel for many
structures), the state exchange and the path read-back: a structure's results
do not depend on its company or on the group it falls into, a refused
structure ends the call after the results before it, and reading a state and a
path in any order, from kept lists or new ones, gives the same numbers."""
import ctypes

import numpy as np
import pytest

import cfneb_inputs as ci
from _cases import gpu_band, lj_structures, perturbed, tersoff_structures

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def g():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2510_16721_gb300 as g
    g.build()
    return g


def _potential(g, pot):
    return {"lj": g.lj_potential, "tersoff": g.tersoff_potential,
            "nep": lambda: g.nep_potential(ci.nep_weights(3), 2.1)}[pot]()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("pot", ["lj", "tersoff", "nep"])
def test_group_equals_single_bitwise(g, pot, precision):
    S = list((lj_structures() if pot == "lj" else tersoff_structures()).values())
    p = _potential(g, pot)
    E, F, V = g.evaluate(S, p, precision)
    for k, s in enumerate(S):
        e, f, v = g.evaluate([s], p, precision)
        assert e[0] == E[k]
        np.testing.assert_array_equal(f[0], F[k])
        np.testing.assert_array_equal(v[0], V[k])


def test_structures_past_the_group_size(g):
    """Two structures of 137,180 atoms do not share a group (2^18 atoms)."""
    R, h = perturbed(*ci.fcc(ci.LJ_A, 35, 35, 28), seed=6, amp=0.03)
    s31 = lj_structures()["vacancy31"]
    E, F, V = g.evaluate([s31, (R, h), (R, h), s31], g.lj_potential(), g.MIXED)
    assert E[1] == E[2] and E[0] == E[3]
    np.testing.assert_array_equal(F[1], F[2])
    np.testing.assert_array_equal(F[0], F[3])
    np.testing.assert_array_equal(V[1], V[2])


def test_refused_structure_ends_the_call(g):
    """The second of three structures is refused (a non-finite coordinate):
    INVALID_ARG, the first one's results written, the others' untouched."""
    S = [lj_structures()["vacancy31"], lj_structures()["triclinic240"],
         lj_structures()["vacancy31"]]
    S[1] = (S[1][0].copy(), S[1][1])
    S[1][0][7, 1] = np.nan
    keep = []
    arr = (g.Structure * 3)(*[g.make_structure(R, h, keep) for R, h in S])
    E = np.full(3, 7.0)
    F = np.full((31 + 240 + 31, 3), 7.0)
    p = g.lj_potential()
    dp = ctypes.POINTER(ctypes.c_double)
    st = g.lib().cfneb_evaluate(arr, 3, ctypes.byref(p), g.FP64, None,
                                E.ctypes.data_as(dp), F.ctypes.data_as(dp), None)
    assert st == g.ERR_INVALID_ARG
    e, f, _ = g.evaluate(S[:1], p, g.FP64)
    assert E[0] == e[0] and np.all(E[1:] == 7.0)
    np.testing.assert_array_equal(F[:31], f[0])
    assert np.all(F[31:] == 7.0)


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("pot", ["lj", "tersoff", "nep"])
def test_state_and_path_in_any_order(g, pot, precision):
    """get_path from the lists the steps kept, again after a state read (the
    same numbers), and from the lists a restored state rebuilds (energies to
    1e-12: other bins round the pair vectors differently)."""
    if pot == "lj":
        R0, h0, R1, h1 = ci.lj_vacancy_hop(ci.LJ_A, (4, 4, 3))
        h1s = ci.strained_cell(h1, 9, 0.005)
        R1, h1, kw = ci.affine(R1, h1, h1s), h1s, dict(k=1.0, dt=0.01)
    else:
        R0, h0, R1, h1 = ci.graphite_hexdiamond_path((4, 3, 2))
        kw = dict(k=0.1, dt=0.02, dt_max=0.02)
    b = gpu_band(g, R0, h0, R1, h1, 6, _potential(g, pot), precision=precision, **kw)
    b.step(7)
    builds = b.list_stats()[0]
    p1 = b.get_path()
    assert b.list_stats()[0] - builds < 4     # some image kept its lists
    st = b.get_state()
    p2 = b.get_path()
    b.set_state(st["X"])
    p3 = b.get_path()
    np.testing.assert_array_equal(p1["positions"], p2["positions"])
    np.testing.assert_array_equal(p1["cells"], p2["cells"])
    np.testing.assert_allclose(p1["energies"], p2["energies"], rtol=1e-12)
    # a restored state carries the lattice rows as c B, rounded at 2^-53 of c:
    # B = X / c + I is off by 2^-53, D by as much, and R = R~ D sums three
    # such terms (and its own roundings) of at most max |R|
    tol = 8.0 * 2.0 ** -53 * max(1.0, np.max(np.abs(p1["positions"])), np.max(np.abs(h0)))
    assert np.max(np.abs(p1["positions"] - p3["positions"])) <= tol
    assert np.max(np.abs(p1["cells"] - p3["cells"])) <= tol
    np.testing.assert_allclose(p1["energies"], p3["energies"], rtol=1e-12)
    assert p1["energies"][0] == p2["energies"][0] and p1["energies"][-1] == p2["energies"][-1]
    np.testing.assert_allclose(p1["positions"][0], R0, atol=2e-5 if precision else 1e-12)


def test_more_structures_than_a_grid_axis_holds(g):
    """66,001 structures in one call, the last of them large enough to take the
    five-pass cell list for all: a kernel's grid holds 65,535 blocks along its
    second and third axes only."""
    pot = g.lj_potential()
    few = [(np.array([[0.1 * k, 0.0, 0.0], [1.05 + 0.11 * k, 0.2, 0.0]]), np.eye(3) * 4.0)
           for k in range(8)]
    R, h = ci.fcc(ci.LJ_A, 20, 20, 18)
    R = R + np.random.default_rng(5).normal(0.0, 0.02, R.shape)
    want = [g.evaluate([s], pot, g.FP64) for s in few + [(R, h)]]
    E, F, V = g.evaluate(few * 8250 + [(R, h)], pot, g.FP64)
    assert np.array_equal(E, np.concatenate([np.tile([w[0][0] for w in want[:8]], 8250), want[8][0]]))
    for k, w in list(enumerate(want[:8])) + [(65528 + j, want[j]) for j in range(8)] + [(66000, want[8])]:
        assert np.array_equal(F[k], w[1][0]) and np.array_equal(V[k], w[2][0])


@pytest.mark.parametrize("reps", [(6, 6, 6), (10, 10, 10)])
@pytest.mark.parametrize("what", ["path", "X", "F", "Fneb"])
def test_read_back_follows_the_stream(g, what, reps):
    """A pinned array whose copy to the device is still queued on the band's stream
    is the target of a read-back: the queued copy gets the array's old bytes."""
    import torch
    R0, h0, R1, h1 = ci.lj_vacancy_hop(reps=reps)
    s = torch.cuda.Stream()
    n, N = len(R0), 5
    opt = g.default_options()
    opt.k_spring, opt.dt, opt.n_max = 1.0, 0.01, N
    band = g.create_band((R0, h0), (R1, h1), N, g.lj_potential(), None, opt, stream=s)
    band.step(1)
    torch.cuda.synchronize()
    size = N * (n if what == "path" else n + 3) * 3
    host = torch.from_numpy(np.random.default_rng(2).uniform(size=size)).pin_memory()
    old, dev = host.clone(), torch.zeros(size, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    with torch.cuda.stream(s):
        torch.cuda._sleep(100000000)  # ~50 ms
        dev.copy_(host, non_blocking=True)
    ptr = ctypes.cast(host.data_ptr(), ctypes.POINTER(ctypes.c_double))
    arg = {k: ptr if k == what else None for k in ("X", "F", "Fneb")}
    if what == "path":
        st = g.lib().cfneb_get_path(band.handle, None, ptr, None, None, None)
    else:
        st = g.lib().cfneb_get_state(band.handle, arg["X"], arg["F"], arg["Fneb"], None, None, None)
    assert st == g.OK
    torch.cuda.synchronize()
    assert torch.equal(dev.cpu(), old)
    want = band.get_path()["positions"] if what == "path" else band.get_state()[what]
    assert np.array_equal(host.numpy(), want.ravel())
    band.destroy()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("reps", [(2, 2, 2), (5, 5, 5), (6, 6, 6), (7, 7, 8)])
def test_state_read_at_once_or_by_array(g, reps, precision):
    """Read-backs converted on the host and on the device (arrays above 96 kB): all
    arrays at once and each by itself are the same values, with zero f_NEB on the end
    images and the lattice rows c B = c I of the end image."""
    R0, h0, R1, h1 = ci.lj_vacancy_hop(reps=reps)
    n, N = len(R0), 5
    band = gpu_band(g, R0, h0, R1, h1, N, g.lj_potential(), k=1.0, dt=0.01, precision=precision)
    band.step(2)
    st = band.get_state()
    for what in ("X", "F", "Fneb"):
        a = np.full((N, n + 3, 3), np.nan)
        arg = {k: g._dptr(a) if k == what else None for k in ("X", "F", "Fneb")}
        assert g.lib().cfneb_get_state(band.handle, arg["X"], arg["F"], arg["Fneb"], None, None,
                                       None) == g.OK
        assert np.array_equal(a, st[what])
    # (B of the initial cell is I to a few roundings, in units of c = n)
    assert np.max(np.abs(st["X"][0, n:] - n * np.eye(3))) <= 1e-14 * n and np.any(st["Fneb"][1])
    assert not np.any(st["Fneb"][[0, -1]])
    band.destroy()
