"""FP64 Tersoff site terms: four lanes per atom in small bands, one thread per
atom in large ones, each with atoms of at most four list entries and with more
(compressed and disordered carbon, a graphite sheet, ragged last tiles), in
single points against the oracle at 1e-10, and the two forms against each
other across the size where the rule switches."""
import numpy as np
import pytest

import cfneb_inputs as ci

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
    if kind == "dense":  # 7% shorter bonds: second neighbours enter the shell
        R, h = 0.86 * R, 0.86 * h
    R = R + rng.normal(0.0, 0.12 if kind == "disordered" else 0.03, R.shape)
    keep = np.sort(rng.permutation(len(R))[:len(R) - drop])
    return R[keep], h


@pytest.mark.parametrize("kind", ["graphite", "diamond", "dense", "disordered"])
@pytest.mark.parametrize("reps,drop", [((1, 1, 1), 0), ((2, 1, 2), 1), ((3, 2, 2), 0),
                                       ((4, 3, 2), 5)])
def test_small_points(g, oracle_mod, kind, reps, drop):
    R, h = _carbon(kind, reps, drop, 3)
    e, Fo, Vo = oracle_mod.Tersoff().evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], g.tersoff_potential(), g.FP64)
    s = max(1.0, np.max(np.abs(Fo)))
    assert abs(E[0] - e.sum()) <= 1e-10 * max(1.0, np.abs(e).sum())
    assert np.max(np.abs(F[0] - Fo)) <= 1e-10 * s
    assert np.max(np.abs(V[0] - Vo)) <= 1e-10 * max(1.0, np.max(np.abs(Vo)))


@pytest.mark.parametrize("kind", ["graphite", "dense", "disordered"])
def test_both_forms_agree(g, kind):
    """The same disordered cell once (lanes) and tiled past the rule's line
    (one thread per atom): per-atom forces agree and the totals scale."""
    R, h = _carbon(kind, (8, 6, 5), 3, 5)
    Rt, ht = ci.tile(R, h, (3, 3, 3))
    assert len(R) < 152 * 2 * 128 <= len(Rt)
    (E1, F1, V1), (E2, F2, V2) = (g.evaluate([s], g.tersoff_potential(), g.FP64)
                                  for s in ((R, h), (Rt, ht)))
    s = max(1.0, np.max(np.abs(F1[0])))
    assert np.max(np.abs(F2[0].reshape(27, -1, 3) - F1[0])) <= 1e-10 * s
    assert abs(E2[0] - 27 * E1[0]) <= 1e-10 * abs(E2[0])
    assert np.max(np.abs(V2[0] - 27 * V1[0])) <= 1e-9 * max(1.0, np.max(np.abs(V2[0])))


@pytest.mark.parametrize("n", [0.01, 0.0125, 0.05, 0.2, 0.25, 0.72751])
@pytest.mark.parametrize("x", [2e-5, 9e-4, 1.1e-3, 0.3])
def test_bond_order_over_n(g, n, x):
    """Three atoms whose bond order is (1 + x)^(-1/2n) with x given (g = 1, one other
    neighbour: zeta = 1): FP64 energy to a few roundings for any n, with x on both
    sides of the series' limit."""
    A, B, l1, l2, r = 1393.6, 346.74, 3.4879, 2.2119, 1.5
    par = [A, B, l1, l2, x ** (1.0 / n), n, 0.0, 1.0, -0.57, 1.95, 0.15]
    R = 5.0 + r * np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [0.5, 0.75 ** 0.5, 0.0]])
    E, F, V = g.evaluate([(R, np.eye(3) * 12.0)], g.tersoff_potential(par), g.FP64)
    d = [np.linalg.norm(R[i] - R[j]) for i, j in ((0, 1), (0, 2), (1, 2))]
    b = np.exp(-np.log1p(par[4] ** n) / (2.0 * n))  # (a beta below 1e-308 is 0: b = 1)
    rep, att = (sum(c * np.exp(-l * v) for v in d) for c, l in ((A, l1), (B, l2)))
    # x ** (1/n) and back: 2^-53 (|log x| + 1) of x, u of that in b
    tol = 1e-14 * (rep + att) * (1.0 + x / (2.0 * n) * abs(np.log(x)))
    assert abs(E[0] - (rep - b * att)) <= tol


@pytest.mark.parametrize("product", [4e37, 8.6e37, 1.2e38, 1.6e38, 1.8e38, 1e39])
def test_large_bond_order_argument(g, oracle_mod, product):
    """Three atoms in the cutoff's edge with (beta zeta)^n zeta about 2^126 to 2^127,
    where FP32 has no normal reciprocal: forces through db/dzeta against the oracle."""
    n, zeta = 50.0, 0.5  # f_C = 1/2 at r = R, g = 1
    beta = (product / zeta) ** (1.0 / n) / zeta
    par = [1393.6, 346.74, 3.4879, 2.2119, beta, n, 0.0, 1.0, -0.57, 1.95, 0.15]
    R = 5.0 + 1.95 * np.array([[0.0, 0.0, 0.0], [1.0, 0.0, 0.0], [0.5, 0.75 ** 0.5, 0.0]])
    h = np.eye(3) * 12.0
    names = ["A", "B", "lambda1", "lambda2", "beta", "n", "c", "d", "h", "R", "D"]
    e, Fo, Vo = oracle_mod.Tersoff(dict(zip(names, par))).evaluate(R, h)
    E, F, V = g.evaluate([(R, h)], g.tersoff_potential(par), g.FP64)
    assert np.max(np.abs(F[0] - Fo)) <= 1e-10 * np.max(np.abs(Fo))
    assert abs(E[0] - e.sum()) <= 1e-10 * abs(e).sum()


def _energy_long(R, h, q):
    """Tersoff energy in long double (the oracle's g, as published, cancels to 1e-8:
    2e-15 of a total)."""
    L = np.longdouble
    rc, W = q["R"] + q["D"], h.astype(L)
    I, D = [], []
    for t in np.ndindex(3, 3, 3):
        d = R[None, :, :] + (np.array(t) - 1) @ h - R[:, None, :]
        i, j = np.nonzero(((d * d).sum(2) < (rc + 0.01) ** 2) & ((d * d).sum(2) > 1e-6))
        I.append(i)
        D.append(R[j].astype(L) + (np.array(t) - 1).astype(L) @ W - R[i].astype(L))
    I, D = np.concatenate(I), np.concatenate(D)
    r = np.sqrt((D * D).sum(1))
    q = {k: L(v) for k, v in q.items()}
    half_pi = 2 * np.arctan(L(1))
    fc = np.where(r < q["R"] - q["D"], L(1), (1 - np.sin(half_pi * (r - q["R"]) / q["D"])) / 2)
    fc = np.where(r < q["R"] + q["D"], fc, L(0))
    E, u = L(0), D / r[:, None]
    for i in range(len(R)):
        e = np.nonzero((I == i) & (fc > 0))[0]
        x = q["h"] - u[e] @ u[e].T
        c2, d2 = q["c"] ** 2, q["d"] ** 2
        z = ((1 + c2 / d2 * x * x / (d2 + x * x)) * (1 - np.eye(len(e)))) @ fc[e]
        b = np.where(z > 0, (1 + (q["beta"] * z) ** q["n"]) ** (-1 / (2 * q["n"])), L(1))
        fr, fa = (q[a] * np.exp(-q[l] * r[e]) for a, l in (("A", "lambda1"), ("B", "lambda2")))
        E += (fc[e] * (fr - b * fa)).sum() / 2
    return E


@pytest.mark.parametrize("kind,reps", [("diamond", (5, 4, 6)), ("graphite", (6, 4, 5)),
                                       ("disordered", (4, 3, 4))])
@pytest.mark.parametrize("images", [0, 84])
def test_total_energy_to_roundings(g, oracle_mod, kind, reps, images):
    """FP64 totals against long double: roundings of single bonds average out, those
    of constants shared by all bonds would not (8e-16 of the total).  Four lanes per
    atom (images = 0: a single point) and, with 84 images, one thread (the end
    image's step energy)."""
    R, h = _carbon(kind, reps, 0, 3)
    want = _energy_long(R, h, oracle_mod.TERSOFF_C1988)
    if images:
        R1 = R.copy()
        R1[0, 0] += 0.1
        o = g.default_options()
        o.n_max = images
        band = g.create_band((R, h), (R1, h), images, g.tersoff_potential(), None, o)
        E = band.image_scalars()["E"][0]
        band.destroy()
    else:
        E = g.evaluate([(R, h)], g.tersoff_potential(), g.FP64)[0][0]
    assert abs(E - want) <= 4e-16 * abs(want)


@pytest.mark.parametrize("lam", [0.01, 0.5, 40.0, 250.0, 300.0, 340.0])
def test_bond_constants_over_exponents(g, oracle_mod, lam):
    """A exp(-lambda1 R) over the exponents that a potential may have: the two-term
    constant (lambda1 R up to 600) and, at the largest, the plain one.  A repulsion's
    exponent is rounded at lambda1 R and lambda1 (r - R), units of up to 663 and 240
    (3e-13 with r's own), and takes lambda1 times the error of r: positions below 16 A
    rounded twice for each atom, 4e-15 A."""
    q = dict(oracle_mod.TERSOFF_C1988)
    q["lambda1"], q["A"] = lam, float(np.exp(lam * 1.45))
    R, h = _carbon("graphite", (3, 3, 2), 0, 3)
    E = g.evaluate([(R, h)], g.tersoff_potential([q[k] for k in q]), g.FP64)[0][0]
    want = _energy_long(R, h, q)
    assert abs(E - want) <= (3e-13 + 4e-15 * lam) * abs(want)
