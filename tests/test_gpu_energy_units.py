"""Dynamic weights in any unit of energy: chi0 scales with its inverse.  Scaling by a power of two is
exact, so a mixed result may move by the rounding of its fixed-point sums alone (2^-45 a term on the
scale the sums are kept at): within the mixed form's 1e-6."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 1e-6}


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("log2", [-40, -20, -10, 10, 20, 40])
@pytest.mark.parametrize("route", ["direct", "kk"])
def test_energy_unit(prec, log2, route):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()

    def run(s):
        n = (6, 5, 7)
        m = wl.random_model(5, wl.SEED_BASE + 95, spread=4.0)
        E, V = m.eig_grid(n)
        q = wl.explicit_q(m, n, (0.21, 0.05, 0.4))
        q.Eq = np.asarray(q.Eq) * s
        W = wl.Workload("units", n, True, 5, 5, E * s, V, wl.fermi_level(E, 2.5) * s, (0, 5), False, [q])
        P = chi0.Plan(W, precision=prec)
        r, i = P.dynamic(np.linspace(0.0, 3.0, 33) * s) if route == "direct" else P.dynamic_kk(9.0 * s, 65)
        P.close()
        return r.cpu().numpy()[0] * s, i.cpu().numpy()[0] * s

    (r0, i0), (r1, i1) = run(1.0), run(2.0**log2)
    assert np.max(np.abs(r1 - r0)) < TOL[prec] * np.max(np.abs(r0))
    assert np.max(np.abs(i1 - i0)) < TOL[prec] * np.max(np.abs(i0))
