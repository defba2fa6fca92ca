"""The arithmetic the weight kernels run, in their sequence (tests/host_math/kernel_math.cpp), against the
FP64 oracle on random, cut and near-degenerate tetrahedra.

Tolerances.  FP64: 1e-11 per tetrahedron static (the oracle comparison of the older host test), 1e-10
dynamic (knots at a frequency carry 2^-53 of D on top, divided by the piece's span, which its volume
pays for).  Mixed: 3e-5 per tetrahedron, 1e-6 on the sum over all of them, as there (not the narrow ones with
frequencies about them: 1/(c - w) takes their midpoint in FP32).  Boxes: the polynomials' truncation, 2.5e-9
(FP32's) and 1e-16 (FP64's), the latter under the moments' rounding, 1e-13."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("kernel_math") / "libkernel_math.so")
    src = os.path.join(HERE, "host_math", "kernel_math.cpp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", src, "-o", out], check=True)
    L = ct.CDLL(out)
    L.host_static.restype = ct.c_double
    L.host_box.restype = ct.c_double
    L.host_box.argtypes = [ct.c_void_p, ct.c_void_p, ct.c_double, ct.c_double, ct.c_double, ct.c_int]
    return L


def p(x):
    return x.ctypes.data_as(ct.c_void_p)


def tetrahedra(kind, n):
    rng = np.random.default_rng(51)
    out = []
    while len(out) < n:
        a = rng.normal(0.0, 1.0, 4)
        b = a + rng.uniform(0.05, 1.5) + rng.normal(0.0, 0.3, 4)
        if kind == "whole":
            a, b = -0.2 - np.abs(a), 0.2 + np.abs(b)
        elif kind == "narrow":  # knots that cluster in pairs and triples
            a = -0.5 + 0.4 * rng.normal() + 10.0 ** rng.uniform(-6, -1) * rng.normal(0.0, 1.0, 4)
            b = a + 0.7 + 10.0 ** rng.uniform(-6, -1) * rng.normal(0.0, 1.0, 4)
        elif kind == "at_ef":  # vertices on either cut plane
            a[rng.integers(0, 4)] = 0.0
            b[rng.integers(0, 4)] = 0.0
        if a.min() < 0.0 and b.max() > 0.0:
            out.append((a, b, rng.uniform(0.1, 1.0, 4)))
    return out


KINDS = ["metal", "whole", "narrow", "at_ef"]


@pytest.mark.parametrize("kind", KINDS)
def test_static_weights(H, oracle_mod, kind):
    s_ref = s_32 = 0.0
    for a, b, f in tetrahedra(kind, 300):
        ref = oracle_mod.tet_integrals(a, b, f)
        g64, g32 = (H.host_static(p(a), p(b), p(f), k) for k in (1, 0))
        assert abs(g64 - ref) <= 1e-11 * abs(ref) + 1e-13, (a, b, f, g64, ref)
        assert abs(g32 - ref) <= 3e-5 * abs(ref) + 1e-9, (a, b, f, g32, ref)
        s_ref += ref
        s_32 += g32
    assert abs(s_32 - s_ref) <= 1e-6 * abs(s_ref)


@pytest.mark.parametrize("kind, fp64", [(k, 1) for k in KINDS] + [(k, 0) for k in KINDS if k != "narrow"])
def test_dynamic_weights(H, oracle_mod, kind, fp64):
    w = np.linspace(0.0, 3.0, 61)
    tol = 1e-10 if fp64 else 3e-5
    tot = np.zeros((4, w.size))
    for a, b, f in tetrahedra(kind, 120):
        rr, ri = oracle_mod.tet_integrals(a, b, f, omega=w)
        gr, gi = np.zeros(w.size), np.zeros(w.size)
        H.host_dynamic(p(a), p(b), p(f), fp64, w.size, p(w), p(gr), p(gi))
        sr = max(np.max(np.abs(rr)), 1e-30)
        assert np.max(np.abs(gr - rr)) <= tol * sr, (a, b, f)
        assert np.max(np.abs(gi - ri)) <= tol * max(np.max(np.abs(ri)), sr), (a, b, f)
        tot += np.stack([rr, ri, gr, gi])
    end = 1e-11 if fp64 else 1e-6
    assert np.max(np.abs(tot[2] - tot[0])) <= end * np.max(np.abs(tot[0]))
    assert np.max(np.abs(tot[3] - tot[1])) <= end * max(np.max(np.abs(tot[1])), np.max(np.abs(tot[0])))


@pytest.mark.parametrize("kind, zmax, tol", [(0, 0.5, 2.5e-9), (1, 2 / 9, 2.5e-9), (2, 5 / 9, 2.5e-9),
                                             (3, 1 / 1.5, 1e-13), (4, 2 / 9, 1e-13), (5, 5 / 9, 1e-13)])
def test_box_polynomials(H, oracle_mod, kind, zmax, tol):
    rng = np.random.default_rng(53)
    for _ in range(300):
        C, R, f = 1.0, rng.uniform(0.1, 0.5), rng.uniform(0.0, 1.0, 4)
        d = np.sort(C + R * rng.uniform(-1.0, 1.0, 4))
        den = rng.choice([-1.0, 1.0]) * R / (zmax * rng.choice([1.0, rng.uniform(0.05, 1.0)]))
        ref = sum(f[j] * oracle_mod.inv_weight(d - (C - den), j) for j in range(4))
        got = H.host_box(p(d), p(f), C, R, den, kind)
        assert abs(got - ref) <= tol * f.sum() / abs(den), (d, f, den, got, ref)
