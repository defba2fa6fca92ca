"""Static weights: groups of q points per launch, units of 4 to 32 tetrahedra, item classes by
index, queues that fill; against the oracle (FP64 1e-12, mixed 1e-6) and, where the arithmetic
is the same, bitwise."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 1e-6}


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


def static(C, W, prec, **kw):
    P = C.Plan(W, precision=prec, **kw)
    out = P.static()
    P.close()
    return out.cpu().numpy() if hasattr(out, "cpu") else out


def close(got, ref, prec):
    return np.max(np.abs(got - ref) / np.max(np.abs(ref))) < TOL[prec]


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n, norb", [((1, 1, 1), 3), ((2, 1, 3), 2), ((5, 7, 3), 4), ((9, 10, 11), 3), ((16, 15, 17), 6)])
def test_units_of_every_size(C, O, prec, n, norb):
    """Odd meshes from one cube up: units that hold the whole mesh, ragged last units."""
    m = wl.random_model(norb, wl.SEED_BASE + 80, spread=4.0)
    E, V = m.eig_grid(n)
    qs = [wl.explicit_q(m, n, q) for q in ((0.21, 0.05, 0.4), (0.5, 0.5, 0.1))]
    W = wl.Workload("units", n, True, norb, norb, E, V, wl.fermi_level(E, norb / 2), (0, norb), False, qs)
    assert close(static(C, W, prec), O.chi0(W), prec)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_groups_do_not_change_results(C, O, prec):
    """35 q (more than one launch takes), shifts, Gamma and explicit data mixed, windows of
    different widths: each value bitwise that of its q alone, and that of a host-input plan, whose
    explicit q points run one at a time."""
    W = wl.tiny_tb(n=6, norb=5, nq=6, seed=wl.SEED_BASE + 81)
    ex = W.qs
    ex[2].window, ex[4].window = (1, 4), (2, 3)
    qs = []
    for j in range(35):
        if j % 6 == 5:
            qs.append(ex[j // 6])
        else:
            s = (j % 6, (j // 6) % 6, (2 * j) % 6)
            qs.append(wl.QPoint(shift=s, gamma=s == (0, 0, 0), window=(0, 5) if j % 4 else (1, 5)))
    W.qs = qs
    got = static(C, W, prec)
    assert close(got, O.chi0(W), prec)
    assert np.array_equal(got, static(C, W, prec, device=False))
    P = C.Plan(W, precision=prec)
    for j in (0, 5, 17, 31, 32, 34):
        one = P.static((C.chi0_q_t * 1)(P.qarr[j])).cpu().numpy()
        assert one[0] == got[j]
    P.close()


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_bands_in_any_order_and_padded_with_nan(C, O, prec):
    """Device energies need not ascend (items are classified by index bounds that hold for any
    order), and bands padded with NaN take no part."""
    W = wl.tiny_tb(n=5, norb=4, nq=0, seed=wl.SEED_BASE + 82)
    W.qs = [wl.QPoint(shift=(1, 2, 3))]
    ref = O.chi0(W)
    p = np.array([2, 0, 3, 1])
    Wp = wl.Workload(W.name, W.n, True, 4, 4, np.ascontiguousarray(W.E[:, p]), np.ascontiguousarray(W.C[:, :, p]), W.ef,
                     (0, 4), False, W.qs)
    assert close(static(C, Wp, prec), ref, prec)
    E = np.concatenate([W.E, np.full((W.ncorner, 2), np.nan)], axis=1)
    V = np.concatenate([W.C, np.zeros((W.ncorner, 4, 2))], axis=2)
    Wn = wl.Workload(W.name, W.n, True, 6, 4, E, V, W.ef, (0, 6), False, W.qs)
    assert close(static(C, Wn, prec), ref, prec)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("case", ["flat", "touching", "tiny_q"])
def test_degenerate_knots(C, O, prec, case):
    """Final tetrahedra whose D coincides at all corners (flat bands), vanishes at vertices (bands
    that touch E_F together) or spans many decades (a free-electron band at small q)."""
    if case == "flat":
        n, nb = (4, 4, 4), 3
        E = np.tile(np.array([-1.0, 0.5, 2.0]), (64, 1))
        U = np.linalg.qr(np.random.default_rng(1).normal(size=(3, 3)))[0].astype(complex)
        V = np.tile(U, (64, 1, 1))
        V[::2] = np.roll(V[::2], 1, axis=1)  # corners alternate along the last axis
        W = wl.Workload("flat", n, True, nb, nb, E, V, 0.0, (0, nb), False, [wl.QPoint(shift=(0, 0, 1))])
    elif case == "touching":
        W = wl.tiny_tb(n=6, norb=2, nq=0, seed=wl.SEED_BASE + 83)
        E = np.sort(np.round(W.E * 2.0) / 2.0, axis=1)  # many corners on few levels
        W = wl.Workload("levels", W.n, True, 2, 2, E, W.C, 0.25, (0, 2), False, [wl.QPoint(shift=(2, 1, 0))])
    else:
        W = wl.free_electron(8, 3, qmax_over_2kf=0.02)
        W.qs = W.qs[1:]
    ref = O.chi0(W)
    assert np.all(np.isfinite(ref)) and close(static(C, W, prec), ref, prec)
