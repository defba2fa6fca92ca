"""q points whose windows lie on both sides of the small overlap kernel's limit (norb x w = 256) in one
call: each value bitwise that of its q alone, whatever it is grouped with."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 1e-6}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("kq", ["shift", "explicit"])
def test_windows_on_both_sides_of_the_limit(oracle_mod, prec, kq):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    n, nb = (3, 4, 3), 17
    m = wl.random_model(nb, wl.SEED_BASE + 90, spread=4.0)
    E, V = m.eig_grid(n)
    windows = [(0, 17), (1, 16), (7, 10), (0, 16), (2, 17), (6, 11), (0, 17), (5, 12)]
    qs = []
    for j, win in enumerate(windows):
        q = wl.explicit_q(m, n, (0.11 + 0.03 * j, 0.2, 0.37)) if kq == "explicit" else wl.QPoint(shift=(j % 3, j % 4, 1))
        q.window = win
        qs.append(q)
    W = wl.Workload("limit", n, True, nb, nb, E, V, wl.fermi_level(E, nb / 2), (0, nb), False, qs)
    P = chi0.Plan(W, precision=prec)
    got = P.static().cpu().numpy()
    one = [P.static((chi0.chi0_q_t * 1)(P.qarr[j])).cpu().numpy()[0] for j in range(len(qs))]
    chi, pairs = P.static_pairs()
    pairs1 = [P.static_pairs((chi0.chi0_q_t * 1)(P.qarr[j]))[1][0] for j in range(len(qs))]
    P.close()
    ref = oracle_mod.chi0(W)
    assert np.max(np.abs(got - ref) / np.max(np.abs(ref))) < TOL[prec]
    assert np.array_equal(got, np.array(one)) and np.array_equal(got, chi)
    assert all(np.array_equal(a, b) for a, b in zip(pairs, pairs1))
