"""Interpolated k+q data: the register forms (up to 10 and 16 orbitals) and the general one at their borders.

Tolerance: a phase is the direction of an overlap <v_0|v_i>, known to norb * eps / m for overlaps of
modulus m or more, and the weighted sum before the normalisation is at least m long (its component on
v_0 is the weighted mean of the overlaps' moduli), so an eigenvector entry is known to 16 norb eps / m^2.
"""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("norb", [1, 9, 10, 11, 16, 17])
def test_interpolated_kq_at_the_borders_of_the_register_forms(norb, oracle_mod):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    W = wl.tiny_tb(n=5, norb=norb, nq=0, seed=wl.SEED_BASE + 70 + norb)
    q = (0.137, 0.261, 0.0831)
    P = chi0.Plan(W, precision="fp64", device=True)
    Eq, Cq = P.interpolate_kq(q)
    P.close()
    Eo, Co = oracle_mod.kq_interpolate(W, q)
    G = np.asarray(W.C).reshape(5, 5, 5, norb, norb)
    m = 1.0
    for s in np.ndindex(3, 3, 3):
        ov = np.einsum("xyzob,xyzob->xyzb", G.conj(), np.roll(G, [i - 1 for i in s], axis=(0, 1, 2)))
        m = min(m, np.abs(ov).min())
    eps = np.finfo(np.float64).eps
    assert np.max(np.abs(Eq - Eo)) <= 1e-12 * np.max(np.abs(Eo))
    assert np.max(np.abs(Cq - Co)) <= 16 * norb * eps / m**2, (np.max(np.abs(Cq - Co)), m)
