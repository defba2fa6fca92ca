"""Cuts between corner levels next to E_F: keys down to the smallest numbers keep their pieces (cut
recipes of the host build; the volumes are those of the same keys at an ordinary scale, to rounding:
the sums of test_static_math.py, 1e-13)."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def H(tmp_path_factory):
    out = str(tmp_path_factory.mktemp("smallest_keys") / "libstatic_math.so")
    src = os.path.join(HERE, "host_math", "static_math.cpp")
    subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", src, "-o", out], check=True)
    return ct.CDLL(out)


@pytest.mark.parametrize("scale", [-1000, -1030, -1060])
def test_pieces_at_every_scale(H, scale):
    rng = np.random.default_rng(41)
    p = lambda x: x.ctypes.data_as(ct.c_void_p)
    got, ref = np.zeros(3), np.zeros(3)
    for _ in range(500):
        a = np.round(rng.uniform(-1.0, 1.0, 4) * 256.0) / 256.0  # exact at every scale here
        D, f = np.abs(a) + 1.0 / 64.0, rng.uniform(0.0, 1.0, 4)
        b, s = a + D, 2.0**scale
        a_s, D_s = a * s, b * s - a * s
        H.host_cut_recipes(p(a), p(D), p(f), p(ref))
        H.host_cut_recipes(p(a_s), p(D_s), p(f), p(got))
        assert abs(got[0] - ref[0]) < 1e-13 and abs(got[1] - ref[1]) < 1e-13, (a, D, got, ref)
