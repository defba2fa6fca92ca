"""Levels exactly at E_F (neither occupied nor empty, as the carving's keys a < 0 and b > 0 have it) at
k, at k+q and at both, against the oracle (FP64 1e-12, mixed 1e-6)."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

TOL = {"fp64": 1e-12, "mixed": 1e-6}


def levels(at, zero):
    W = wl.tiny_tb(n=6, norb=4, nq=2, seed=wl.SEED_BASE + 121)
    for Q in W.qs:
        Q.Eq = np.array(Q.Eq) - W.ef
    W.E = np.array(W.E) - W.ef
    W.ef = 0.0
    for E, here, step in [(W.E, at != "kq", 5)] + [(Q.Eq, at != "k", 7) for Q in W.qs]:
        if here:
            for c in range(0, E.shape[0], step):
                E[c, np.argmin(np.abs(E[c]))] = zero
    return W


@pytest.mark.parametrize("prec", ["fp64", "mixed"])
@pytest.mark.parametrize("at", ["k", "kq", "both"])
@pytest.mark.parametrize("zero", [0.0, -0.0])
def test_levels_at_the_fermi_level_match_the_oracle(oracle_mod, prec, at, zero):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    W = levels(at, zero)
    assert (W.E == 0.0).any() == (at != "kq") and all((Q.Eq == 0.0).any() == (at != "k") for Q in W.qs)
    omega = np.linspace(0.05, 3.0, 17)
    ref = oracle_mod.chi0(W)
    dyn = [oracle_mod.chi0_q(W, Q, omega=omega) for Q in W.qs]
    P = chi0.Plan(W, precision=prec)
    got = P.static().cpu().numpy()
    re, im = (x.cpu().numpy() for x in P.dynamic(omega))
    P.close()
    assert np.max(np.abs(got - ref)) < TOL[prec] * np.max(np.abs(ref)), (got, ref)
    for j, (r, i) in enumerate(dyn):
        assert np.max(np.abs(re[j] - r)) < TOL[prec] * np.max(np.abs(r))
        assert np.max(np.abs(im[j] - i)) < TOL[prec] * np.max(np.abs(i))
