"""Dynamic weights where a band pair's D is constant over a tetrahedron and a frequency meets it,
against the oracle (FP64 1e-12, mixed 1e-6, normwise per q).

The levels are dyadic, so that D and w are exact in both precisions: at w = D the pole's own term is
dropped (its principal value) and what is left is an ordinary number."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 1e-6}
PRECS = ["fp64", "mixed"]


@pytest.fixture(scope="module")
def C():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    return chi0


@pytest.fixture(scope="module")
def O(oracle_mod):
    return oracle_mod


def run(C, W, prec, omega):
    P = C.Plan(W, precision=prec)
    re, im = P.dynamic(omega)
    P.close()
    return re.cpu().numpy()[0], im.cpu().numpy()[0]


def flat(n=(4, 4, 4)):
    """Three flat bands, D = 1.5 and 3 for every pair of corners."""
    nc = int(np.prod(n))
    U = np.linalg.qr(np.random.default_rng(1).normal(size=(3, 3)))[0].astype(complex)
    V = np.tile(U, (nc, 1, 1))
    V[::2] = np.roll(V[::2], 1, axis=1)  # corners alternate along the last axis
    return wl.Workload("flat", n, True, 3, 3, np.tile([-1.0, 0.5, 2.0], (nc, 1)), V, 0.0, (0, 3), False,
                       [wl.QPoint(shift=(0, 0, 1))])


def split():
    """A band and the same 1/2 higher, cut by the Fermi surface, and two empty ones far above, at Gamma:
    D = 1/2 at every k for the lower two."""
    n = (4, 4, 4)
    E, _ = wl.random_model(2, wl.SEED_BASE + 1, spread=1.0).eig_grid(n)
    E = np.round((E - E.mean(axis=0)) * 2.0**16) / 2.0**16
    E = np.stack([E[:, 0], E[:, 0] + 0.5, E[:, 1] + 3.0, E[:, 1] + 3.5], axis=1)
    return wl.Workload("split", n, True, 4, 4, E, None, wl.fermi_level(E, 0.7), (0, 4), True,
                       [wl.QPoint(shift=(0, 0, 0), gamma=True)])


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("n", [(1, 1, 2), (4, 4, 4)])
@pytest.mark.parametrize("omega", [np.arange(33) / 8.0, np.array([1.5]), np.array([-3.0, 0.0, 1.25])],
                         ids=["grid", "single", "few"])
def test_flat_bands_with_a_frequency_on_them(C, O, prec, n, omega):
    W = flat(n)
    r, i = O.chi0_q(W, W.qs[0], omega=omega)
    gr, gi = run(C, W, prec, omega)
    assert np.max(np.abs(gr - r)) < TOL[prec] * max(np.max(np.abs(r)), 1e-300), (gr, r)
    assert np.all(i == 0.0) and np.all(gi == 0.0)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("ntet", [1, 2, 3])
def test_a_few_flat_tetrahedra(C, O, prec, ntet):
    """An even and an odd number of pieces on the pole (what is wrong in each may cancel in pairs)."""
    W = flat()
    tet, vol = wl.builtin_tetra(W.n, np.arange(7, 7 + ntet))
    omega = np.array([0.25, 1.5, 3.0])
    r, _ = O.chi0_q(W, W.qs[0], omega=omega, tet=tet, tvol=vol)
    P = C.Plan(W, precision=prec, tetra=(tet, vol))
    gr, gi = (x.cpu().numpy()[0] for x in P.dynamic(omega))
    P.close()
    assert np.max(np.abs(gr - r)) < TOL[prec] * np.max(np.abs(r)) and np.all(gi == 0.0), (gr, r)


@pytest.mark.parametrize("prec", PRECS)
def test_bands_split_rigidly_at_gamma(C, O, prec):
    """The value on the pole against the mean of the oracle's on both sides of it, where the pole's
    terms cancel: what is left is even in the distance h, so two distances give its error."""
    W = split()
    omega = np.arange(25) / 8.0
    h = 2.0**-7
    sides = np.array([0.5 - 2 * h, 0.5 - h, 0.5 + h, 0.5 + 2 * h])
    r, i = O.chi0_q(W, W.qs[0], omega=omega)
    s, _ = O.chi0_q(W, W.qs[0], omega=sides)
    gr, gi = run(C, W, prec, omega)
    at = int(np.flatnonzero(omega == 0.5)[0])
    near, far = 0.5 * (s[1] + s[2]), 0.5 * (s[0] + s[3])
    assert abs(gr[at] - near) <= 2.0 * abs(near - far), (gr[at], near, far)
    off = np.arange(len(omega)) != at
    assert np.max(np.abs(gr - r)[off]) < TOL[prec] * np.max(np.abs(r[off]))
    assert np.max(np.abs(gi - i)[off]) < TOL[prec] * np.max(np.abs(i))


def mixed_spectrum():
    """Flat bands D = 1.5 and 3 beside a dispersive one that covers the same range."""
    W = flat()
    c = wl.corner_frac(W.n, True)
    E = np.array(W.E)
    E[:, 2] = 1.5 + np.round(1.25 * np.cos(2 * np.pi * c).mean(axis=1) * 2.0**16) / 2.0**16
    return wl.Workload("beside", W.n, True, 3, 3, E, W.C, 0.0, (0, 3), False, W.qs)


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("extra", ["signs", "three", "eight", "close"])
def test_repeats_at_a_flat_band_leave_the_others_alone(C, O, prec, extra):
    """The same frequency several times (and with the other sign, and as neighbours that one FP32 number
    stands for) where a flat D equals it: every other frequency keeps its values, bitwise in the mixed
    form (integer sums), and all of Im agrees with the oracle."""
    W = mixed_spectrum()
    omega = np.arange(1, 33) / 8.0
    more = {"signs": [-1.5], "three": [1.5, 1.5], "eight": [1.5] * 4 + [-1.5] * 3,
            "close": 1.5 + 1e-9 * np.arange(1, 8)}[extra]
    all_w = np.concatenate([omega, more])
    r0, i0 = run(C, W, prec, omega)
    r1, i1 = run(C, W, prec, all_w)
    _, i = O.chi0_q(W, W.qs[0], omega=all_w)
    assert np.max(np.abs(i1 - i)) < TOL[prec] * np.max(np.abs(i)), (i1, i)
    n = len(omega)
    if prec == "mixed":
        assert np.array_equal(r1[:n], r0) and np.array_equal(i1[:n], i0)
    else:
        assert np.max(np.abs(r1[:n] - r0)) < TOL[prec] * np.max(np.abs(r0))
        assert np.max(np.abs(i1[:n] - i0)) < TOL[prec] * np.max(np.abs(i0))


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("odd", [[np.nan], [np.nan, np.inf, -np.inf, np.nan, 1e300], [np.nan] * 40, [np.inf] * 3],
                         ids=["nan", "mixture", "many_nan", "inf"])
def test_frequencies_that_are_not_finite_stay_by_themselves(C, prec, odd):
    """The finite frequencies keep their values (bitwise in the mixed form); a NaN has Re = NaN and
    Im = 0, an infinite one (in the mixed form one past FP32's range) the limit 0."""
    W = mixed_spectrum()
    omega = np.arange(1, 33) / 8.0 + 0.03
    rng = np.random.default_rng(7)
    all_w = np.concatenate([omega, odd])
    order = rng.permutation(len(all_w))
    r0, i0 = run(C, W, prec, omega)
    r1, i1 = np.empty(len(all_w)), np.empty(len(all_w))
    r1[order], i1[order] = run(C, W, prec, all_w[order])
    n = len(omega)
    if prec == "mixed":
        assert np.array_equal(r1[:n], r0) and np.array_equal(i1[:n], i0)
    else:
        assert np.max(np.abs(r1[:n] - r0)) < TOL[prec] * np.max(np.abs(r0))
        assert np.max(np.abs(i1[:n] - i0)) < TOL[prec] * np.max(np.abs(i0))
    nan = np.isnan(all_w[n:])
    assert np.all(np.isnan(r1[n:][nan]))
    assert np.all(np.abs(r1[n:][~nan]) <= 1e-290) and np.all(i1[n:] == 0.0)


@pytest.mark.parametrize("prec", PRECS)
def test_no_finite_frequency_at_all(C, prec):
    r, i = run(C, flat(), prec, np.array([np.nan, np.inf]))
    assert np.isnan(r[0]) and r[1] == 0.0 and np.all(i == 0.0)
