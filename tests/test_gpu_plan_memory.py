"""Device memory a plan holds."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

MB = 1 << 20


@pytest.fixture(scope="module")
def C():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    W = wl.tiny_tb(n=2, norb=2, nq=1)
    chi0.Plan(W, precision="fp64").static().cpu()  # (the context's own allocations)
    return chi0


def free_bytes():
    import torch
    torch.cuda.synchronize()
    return torch.cuda.mem_get_info()[0]


def test_small_fp64_plan(C):
    """A 6^3 mesh of four bands: its data are a few hundred KB; the rest is the dynamic weights'
    per-warp scratch (some 152 x 4 x 2 warps, 160 MB at most)."""
    W = wl.tiny_tb(n=6, norb=4, nq=1)
    S = C.DeviceInputs(W)
    f0 = free_bytes()
    P = C.Plan(W, precision="fp64", staged=S)
    held = f0 - free_bytes()
    P.close()
    assert held < 180 * MB, held / MB


def test_band_pair_totals_of_a_wide_window(C):
    """1024 bands without matrix elements, 8 q: the fixed-point totals of the q in flight stay within
    64 MB (8 MB a q), and each q's block is bitwise that of the q alone."""
    nb = 1024
    E = np.linspace(-1.0, 1.0, nb)[None, :] * np.array([1.0, 1.1])[:, None]
    W = wl.Workload("wide", (1, 1, 2), True, nb, nb, E, None, 0.0, (0, nb), True,
                    [wl.QPoint(shift=(0, 0, 1)) for _ in range(8)])
    q = [wl.QPoint(shift=(0, 0, 1), window=(0, nb) if j % 2 else (8 * j, nb)) for j in range(12)]
    W.qs = q
    S = C.DeviceInputs(W)
    P = C.Plan(W, precision="fp64", staged=S)
    f0 = free_bytes()
    import torch
    npairs = sum((nb - (0 if j % 2 else 8 * j)) ** 2 for j in range(12))
    chi = torch.empty(12, dtype=torch.float64, device="cuda")
    pairs = torch.empty(npairs, dtype=torch.float64, device="cuda")
    f0 = free_bytes()
    C.chi0_static_pairs(P.h, P.qarr, 12, chi.data_ptr(), pairs.data_ptr())
    held = f0 - free_bytes()
    assert held <= 96 * MB, held / MB
    off = 0
    for j in range(12):
        w = nb - (0 if j % 2 else 8 * j)
        one, p1 = torch.empty(1, dtype=torch.float64, device="cuda"), torch.empty(w * w, dtype=torch.float64, device="cuda")
        C.chi0_static_pairs(P.h, (C.chi0_q_t * 1)(P.qarr[j]), 1, one.data_ptr(), p1.data_ptr())
        assert torch.equal(p1, pairs[off:off + w * w]) and torch.equal(one, chi[j:j + 1])
        off += w * w
    P.close()
