"""Mixed dynamic weights of a window that also holds bands far from the others (core levels, placeholders
for missing bands): the sums of the ordinary bands keep their range and rounding, against the oracle.
The far bands' pairs add |M|^2 / 10^4 and less, so the result is that of the ordinary bands, and the
mixed form's 1e-6 holds."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("cma", [True, False])
@pytest.mark.parametrize("far", [(1e4,), (1e7, 1e7), (1e10,), (1e15,), (-1e4,), (-1e4, 1e6), (-1e10, 1e12)])
def test_far_bands(oracle_mod, far, cma):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    n, norb = (6, 5, 7), 5
    nc = int(np.prod(n))
    E, V = wl.random_model(norb, wl.SEED_BASE + 96, spread=4.0).eig_grid(n)
    ef = wl.fermi_level(E, 2.5)
    below = [x for x in far if x < 0]
    above = [x for x in far if x > 0]
    nb = norb + len(far)
    Ef = np.concatenate([np.full((nc, len(below)), below), E, np.full((nc, len(above)), above)], axis=1)
    U = np.zeros((nc, norb, nb), dtype=complex)
    U[:, :, len(below):len(below) + norb] = V
    U[:, 0, :len(below)] = 1.0
    U[:, -1, len(below) + norb:] = 1.0
    W = wl.Workload("far", n, True, nb, norb, Ef, None if cma else U, ef, (0, nb), cma, [wl.QPoint(shift=(2, 1, 3))])
    om = np.linspace(0.0, 6.0, 41)
    r0, i0 = oracle_mod.chi0_q(W, W.qs[0], omega=om)
    P = chi0.Plan(W, precision="mixed")
    r1, i1 = P.dynamic(om)
    P.close()
    r1, i1 = r1.cpu().numpy()[0], i1.cpu().numpy()[0]
    assert np.max(np.abs(r1 - r0)) < 1e-6 * np.max(np.abs(r0))
    assert np.max(np.abs(i1 - i0)) < 1e-6 * np.max(np.abs(i0))
