"""The FP32 series never reads past its coefficients (array bounds checked in a host build), also
where no convergence test ends it."""
import os
import subprocess

HERE = os.path.dirname(os.path.abspath(__file__))


def test_series_stay_inside_their_tables(tmp_path):
    out = str(tmp_path / "series_bounds")
    src = os.path.join(HERE, "host_math", "series_bounds.cpp")
    subprocess.run(["g++", "-O1", "-std=c++17", "-fsanitize=bounds", "-fsanitize-undefined-trap-on-error", src, "-o", out],
                   check=True)
    r = subprocess.run([out], capture_output=True, text=True)
    assert r.returncode == 0, r
    v = [float(x) for x in r.stdout.split()]
    assert abs(v[0] - v[1]) <= 1e-5 * abs(v[1]) and v[2] == v[3] == 0.0
