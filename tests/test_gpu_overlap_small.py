"""Overlaps of small blocks: 3 x 3 tiles at every remainder, one to several corners a step, more tiles
than lanes, the general form past the border, against the oracle (FP64 1e-12, mixed 1e-6, normwise).
5^3 corners: the last step of a warp is ragged for every number of corners a step."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec, tol", [("fp64", 1e-12), ("mixed", 1e-6)])
@pytest.mark.parametrize("explicit, c64", [(True, False), (True, True), (False, False)])
@pytest.mark.parametrize("norb", [2, 3, 4, 7, 9, 10, 15, 16, 17])
def test_overlap_blocks_of_every_size(norb, explicit, c64, prec, tol, oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    W = wl.tiny_tb(n=5, norb=norb, nq=2 if explicit else 0, seed=wl.SEED_BASE + 90 + norb, explicit=explicit,
                   cdtype=np.complex64 if c64 else np.complex128)
    if not explicit:
        W.qs = [wl.QPoint(shift=(1, 0, 2)), wl.QPoint(shift=(2, 3, 1))]
    P = chi0.Plan(W, precision=prec, device=True)
    got = np.asarray(P.static().cpu(), dtype=np.float64)
    P.close()
    ref = np.asarray(oracle_mod.chi0(W), dtype=np.float64)
    assert np.max(np.abs(got - ref) / np.abs(ref)) <= tol, (got, ref)
