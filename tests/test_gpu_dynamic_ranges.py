"""Dynamic weights: frequencies in any order and count, boxes of every kind, units of one to 32
tetrahedra, against the oracle (FP64 1e-12, mixed 1e-6, normwise per q)."""
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


def run(C, W, prec, omega):
    P = C.Plan(W, precision=prec)
    re, im = P.dynamic(omega)
    P.close()
    return re.cpu().numpy(), im.cpu().numpy()


def err(got, ref):
    return np.max(np.max(np.abs(got - ref), axis=1) / np.maximum(np.max(np.abs(ref), axis=1), 1e-300))


def model(n, norb, seed, spread=4.0):
    m = wl.random_model(norb, wl.SEED_BASE + seed, spread=spread)
    E, V = m.eig_grid(n)
    qs = [wl.explicit_q(m, n, q) for q in ((0.21, 0.05, 0.4),)]
    return wl.Workload("ranges", n, True, norb, norb, E, V, wl.fermi_level(E, norb / 2), (0, norb), False, qs)


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("grid", ["one", "seven", "eight", "unsorted_signed", "repeated", "spread", "full", "two_passes"])
def test_frequency_grids(C, O, prec, grid):
    """A single frequency to two passes; any order, signs and repeats; a range over five decades; one
    pass of exactly 256."""
    rng = np.random.default_rng(31)
    omega = {"one": [1.3], "seven": np.linspace(0.1, 3.0, 7), "eight": np.linspace(0.1, 3.0, 8),
             "unsorted_signed": rng.permutation(np.concatenate([np.linspace(0.0, 3.0, 31), -np.linspace(0.05, 2.0, 18)])),
             "repeated": np.repeat([0.0, 0.7, -0.7, 2.1], 5), "spread": np.geomspace(1e-4, 30.0, 40),
             "full": np.linspace(0.0, 2.0, 256), "two_passes": np.linspace(0.0, 2.0, 259)}[grid]
    omega = np.asarray(omega, dtype=np.float64)
    W = model((5, 4, 6), 4, 84)
    r, i = O.chi0_q(W, W.qs[0], omega=omega)
    gr, gi = run(C, W, prec, omega)
    # (a grid outside the spectrum has Im = 0: compared on the scale of Re)
    scale = max(np.max(np.abs(i)), 1e-3 * np.max(np.abs(r)))
    assert err(gr, r[None, :]) < TOL[prec]
    assert np.max(np.abs(gi[0] - i)) < TOL[prec] * scale


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("n, norb, wmax", [((1, 1, 1), 2, 3.0), ((3, 2, 2), 12, 1.0), ((4, 4, 4), 5, 0.05),
                                           ((6, 5, 7), 3, 8.0), ((13, 12, 11), 4, 0.8)])
def test_meshes_and_boxes(C, O, prec, n, norb, wmax):
    """Pieces in every kind of box: frequencies far below the spectrum (geometric and wide boxes),
    across it (fine boxes, unboxed pieces on coarse meshes) and past it."""
    if n == (1, 1, 1) and prec == "mixed":
        pytest.skip("one k point: flat bands, whose pole 1/(D - w) magnifies the FP32 rounding of D")
    W = model(n, norb, 85 + norb)
    omega = np.linspace(0.0, wmax, 33)
    r, i = O.chi0_q(W, W.qs[0], omega=omega)
    gr, gi = run(C, W, prec, omega)
    assert err(gr, r[None, :]) < TOL[prec]
    assert np.max(np.abs(gi[0] - i)) < TOL[prec] * max(np.max(np.abs(i)), 1e-3 * np.max(np.abs(r)))
