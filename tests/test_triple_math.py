"""FP32 entries of three clustered knots against the per-vertex table in FP64, on the CPU.

Tolerance, in units of max f / s (s the largest knot): the entries are formed by four differences
divided by the gaps to the fourth knot, each with some ten roundings of 2^-24 on either side, so
20 x 2^-24 / gap^4, gap in units of s: at least 0.46 for the knots of a near pair (the frequency lies
within two half-widths of the piece), at least 0.2 for any knots the form takes."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("triple_math") / "libtriple_math.so")
    src = os.path.join(HERE, "host_math", "triple_math.cpp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", src, "-o", out], check=True)
    return ct.CDLL(out)


@pytest.mark.parametrize("sign", [1.0, -1.0])
@pytest.mark.parametrize("where", ["top", "bottom", "close"])
@pytest.mark.parametrize("ties", ["none", "two", "three"])
def test_triple_entries_match_the_table(H, sign, where, ties):
    rng = np.random.default_rng(31)
    out = np.zeros(2)
    gap = 0.2 if where == "close" else 0.46
    took = 0
    for i in range(2000):
        w = 0.25 * rng.uniform() ** (1 + i % 8)  # spread of the cluster, down to a few roundings
        c = np.array([1.0, 1.0 - w * rng.uniform(), 1.0 - w])
        if ties == "two":
            c[1] = c[rng.choice([0, 2])]
        elif ties == "three":
            c[:] = 1.0
        if where == "top":
            a = rng.uniform(-1.0, 1.0 / 3.0) if i % 50 else 0.0
        elif where == "bottom":
            c *= rng.uniform(0.01, 0.4)
            a = rng.choice([-1.0, 1.0])
        else:
            a = rng.uniform(0.3, 0.8)
        x = np.sort(sign * rng.uniform(0.1, 9.0) * np.append(c, a)).astype(np.float32)
        f = rng.uniform(0.0, 1.0, 4).astype(np.float32)
        s = float(np.abs(x).max())
        if not H.host_triple_table(x.ctypes.data_as(ct.c_void_p), f.ctypes.data_as(ct.c_void_p),
                                   out.ctypes.data_as(ct.c_void_p)):
            continue
        took += 1
        assert abs(out[0] - out[1]) * s <= 20 * 2.0**-24 / gap**4, (x, f, out)
    assert took > (200 if where == "close" else 1500), took
