"""FP64 weights of a band whose corner levels at k are closer to E_F than 2^-1022, on either side of it (the
other bands keep a gap, so that no final tetrahedron has D near 0): the cuts depend on the levels' ratios
alone, so the results are those of levels at 1e-290, to 1e-12."""
import numpy as np
import pytest

from paper_1407_3444_gb300 import workloads as wl

pytestmark = pytest.mark.gpu


def workload(tiny):
    W = wl.tiny_tb(n=5, norb=3, nq=2, seed=wl.SEED_BASE + 122)
    E = np.sort(-np.abs(W.E - W.ef) - 0.3, axis=1)
    E[:, 2] = np.array([-1.0, 2.0, -3.0, 4.0, 5.0, -6.0, 7.0])[np.arange(E.shape[0]) % 7] * tiny
    for Q in W.qs:
        Q.Eq = np.sort(np.abs(np.asarray(Q.Eq) - W.ef) + 0.3, axis=1)
    W.E, W.ef = E, 0.0
    return W


@pytest.mark.parametrize("tiny", [1e-309, 5e-324])
def test_the_smallest_levels_keep_their_pieces(oracle_mod, tiny):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    out = []
    for scale in (tiny, 1e-290):
        P = chi0.Plan(workload(scale), precision="fp64")
        out.append([P.static().cpu().numpy()] + [x.cpu().numpy() for x in P.dynamic(np.linspace(0.05, 3.0, 17))])
        P.close()
    W = workload(1e-100)
    assert np.max(np.abs(out[1][0] - oracle_mod.chi0(W))) <= 1e-12 * np.max(np.abs(out[1][0]))
    for got, ref in zip(*out):
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref)), (got, ref)


@pytest.mark.parametrize("tiny", [4e-309, 1e-308, 5e-324])
def test_pieces_narrower_than_the_normal_range(tiny):
    """Two flat-to-rounding bands that touch E_F from either side (D below 2^-1022): past D the terms
    1/(D - w) + 1/(D + w) cancel, so that band pair adds nothing to the others' Re and Im."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1407_3444_gb300 import build, chi0
    build.build()
    chi0.lib()
    omega = np.linspace(0.05, 3.0, 17)

    def run(scale):
        W = wl.tiny_tb(n=5, norb=3, nq=1, seed=wl.SEED_BASE + 123)
        k = 1.0 + np.arange(W.ncorner) % 5
        W.E = np.sort(-np.abs(W.E - W.ef) - 0.3, axis=1)
        W.E[:, 2] = -scale * k
        Q = W.qs[0]
        Q.Eq = np.sort(np.abs(np.asarray(Q.Eq) - W.ef) + 0.3, axis=1)
        Q.Eq[:, 0] = scale * k
        W.ef = 0.0
        P = chi0.Plan(W, precision="fp64")
        out = [x.cpu().numpy() for x in P.dynamic(omega)]
        P.close()
        return out

    for got, ref in zip(run(tiny), run(1e-30)):
        assert np.max(np.abs(got - ref)) <= 1e-12 * np.max(np.abs(ref)), (got, ref)
