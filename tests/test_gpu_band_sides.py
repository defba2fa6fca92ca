"""Which side of eF a level lies on, at the ends of the number range: a level at eF (of either zero
sign) is on neither side, the smallest number off it is on one.  The results are compared with each
other: both zeros bitwise, the smallest numbers with 1e-300 of the same sign to 1e-12 (the cut
fractions of both are 0 to rounding)."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def static(level, prec):
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    W = wl.tiny_tb(n=4, norb=3, nq=2, seed=wl.SEED_BASE + 120)
    for Q in W.qs:
        Q.Eq = np.array(Q.Eq) - W.ef
    W.E = np.array(W.E) - W.ef
    W.ef = 0.0
    E = W.E.reshape(-1, 3)
    for c in range(0, E.shape[0], 5):
        E[c, np.argmin(np.abs(E[c]))] = level
    P = chi0.Plan(W, precision=prec, device=True)
    out = P.static().cpu().numpy()
    P.close()
    return out


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
def test_levels_at_the_fermi_level(prec):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    assert np.array_equal(static(0.0, prec), static(-0.0, prec))


@pytest.mark.parametrize("sign", [1.0, -1.0])
def test_the_smallest_levels_have_a_side(sign):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    got, ref = static(sign * 5e-324, "fp64"), static(sign * 1e-300, "fp64")
    assert np.max(np.abs(got - ref) / np.abs(ref)) <= 1e-12, (got, ref)
