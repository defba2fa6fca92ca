"""The static weights' own arithmetic (tests/host_math/static_math.cpp) on the CPU: cut recipes
against cut_piece, the FP64 series about the mean against an extended-precision sum, the FP32
short recurrence against series_sum.

Tolerances.  Cuts: sums of at most 9 products of some 20 roundings of numbers up to 2: 1e-13.
Mean series: a dozen roundings at the end and offsets exact to one each, amplified by at most
(1 + R)/(1 - R) = 8.1 at the widest tier: 12 x 8.1 x 2^-53 = 1.1e-14; below R = 0.3 the factor is
1.9: 2.6e-15.  Short recurrence: both forms carry some ten roundings of 2^-24, amplified by
(1 + r)/(1 - r) = 5.7 at r = 0.7: 10 x 5.7 x 2^-24 = 3.4e-6; their mean difference, which the
common truncation rule keeps from being a bias, over N samples below that over sqrt(N).
Triple clusters: sums of terms of size f/s (s the largest knot) divided by gaps of at least s/9
to the fourth knot three times over: 9^3 x 20 roundings x 2^-53 = 1.6e-12 of f/s."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("static_math") / "libstatic_math.so")
    src = os.path.join(HERE, "host_math", "static_math.cpp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", src, "-o", out], check=True)
    return ct.CDLL(out)


def _p(x):
    return x.ctypes.data_as(ct.c_void_p)


@pytest.mark.parametrize("kind", ["metal", "gapped", "zero_keys", "inverted"])
def test_cut_recipes_match_cut_piece(H, kind):
    rng = np.random.default_rng(21)
    a1, a2 = np.zeros(3), np.zeros(3)
    seen = set()
    for _ in range(4000):
        a = rng.uniform(-1.0, 1.0, 4)
        D = rng.uniform(0.0, 1.5, 4)
        if kind == "gapped":
            D += 1.5
        elif kind == "zero_keys":  # vertices on either cut plane, and D = 0
            a[rng.integers(0, 4)] = 0.0
            D[rng.integers(0, 4)] = 0.0
        elif kind == "inverted":
            D -= 0.6
        f = rng.uniform(0.0, 1.0, 4)
        H.host_cut_recipes(_p(a), _p(D), _p(f), _p(a1))
        H.host_cut_pieces(_p(a), _p(D), _p(f), _p(a2))
        assert np.max(np.abs(a1 - a2)) < 1e-13, (a, D, f, a1, a2)
        seen.add((int((a < 0).sum()), int((a + D > 0).sum())))
    assert len(seen) >= (5 if kind == "gapped" else 8), seen  # (a + D > 0 throughout: five cases)


@pytest.mark.parametrize("spread, tol", [(1e-9, 2.6e-15), (1e-4, 2.6e-15), (0.01, 2.6e-15), (0.07, 2.6e-15),
                                         (0.2, 2.6e-15), (0.6, 1.1e-14), (0.78, 1.1e-14)])
def test_mean_series_every_tier(H, spread, tol):
    rng = np.random.default_rng(22)
    v = ct.c_double()
    ld = np.longdouble
    used = set()
    for _ in range(300):
        d = rng.uniform(0.3, 7.0) * (1.0 + spread * rng.uniform(-1.0, 1.0, 4))
        f = rng.uniform(0.0, 1.0, 4)
        tier = H.host_mean_series(_p(d), _p(f), ct.byref(v))
        c = ld(d.astype(ld).mean())
        e = (d.astype(ld) - c) / c
        if tier < 0:
            assert float(np.max(np.abs(e))) > 0.78
            continue
        used.add(tier)
        h, p, s = np.ones(4, dtype=ld), np.ones(4, dtype=ld), ld(0.25) * f.astype(ld).sum()
        for k in range(1, 260):
            h[0] = e[0] * h[0]
            for i in range(1, 4):
                h[i] = h[i - 1] + e[i] * h[i]
            p = h[3] + e * p
            s += ld((-1) ** k * 6) / ld((k + 1) * (k + 2) * (k + 3) * (k + 4)) * (f.astype(ld) * p).sum()
        ref = s / c
        assert abs(float((ld(v.value) - ref) / ref)) < tol, (tier, d, f, v.value, ref)
    assert used


def test_mean_series_leaves_knots_with_zeros(H):
    v = ct.c_double()
    f = np.ones(4)
    for d in ([0.0, 0.0, 0.0, 0.0], [0.0, 1.0, 1.0, 1.0], [0.0, 0.0, 0.0, 1.0]):
        assert H.host_mean_series(_p(np.array(d)), _p(f), ct.byref(v)) == -1


@pytest.mark.parametrize("spread", [0.003, 0.05, 0.2, 0.5, 0.7])
def test_short_recurrence_is_series_sum(H, spread):
    rng = np.random.default_rng(23)
    v, w = ct.c_float(), ct.c_float()
    diff = []
    for _ in range(4000):
        d = np.sort((rng.uniform(0.5, 4.5) * (1.0 + spread * rng.uniform(-1.0, 1.0, 4))).astype(np.float32))
        f = rng.uniform(0.0, 1.0, 4).astype(np.float32)
        if H.host_short_series(_p(d), _p(f), ct.byref(v), ct.byref(w)):
            diff.append((v.value - w.value) / w.value)
    diff = np.array(diff)
    assert len(diff) > 1000 and np.max(np.abs(diff)) < 3.4e-6
    assert abs(diff.mean()) < 3.4e-6 / np.sqrt(len(diff))


@pytest.mark.parametrize("width", [0.0, 1e-14, 1e-9, 1e-4, 0.02, 0.06])
@pytest.mark.parametrize("where", ["apart", "zero", "near"])
def test_triple_cluster_matches_the_table(H, width, where):
    rng = np.random.default_rng(24)
    v, w = ct.c_double(), ct.c_double()
    done = 0
    for _ in range(400):
        c = rng.choice([-1.0, 1.0]) * rng.uniform(0.2, 2.0)
        a = {"apart": rng.uniform(-3.0, 3.0), "zero": 0.0, "near": c * rng.choice([0.6, 1.6])}[where]
        x = np.sort(np.concatenate([c * (1.0 + width * rng.uniform(-1.0, 1.0, 3)), [a]]))
        f = rng.uniform(0.0, 1.0, 4)
        if not H.host_triple(_p(x), _p(f), ct.byref(v), ct.byref(w)):
            assert abs(a - c) < 0.3 * abs(c)  # all four together: not this case
            continue
        done += 1
        assert abs(v.value - w.value) < 1.6e-12 * f.sum() / np.max(np.abs(x)), (x, f, v.value, w.value)
    assert done > 250
