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
