"""The bench's roofline of the FP32-class Laplacian product counts each pipe's operations: features on the integer pipe
are no FP32 operations, and which features those are follows the library's rule."""
import math
import os
import re
import sys

import numpy as np

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
sys.path.insert(0, ROOT)


def test_operations_are_counted_per_pipe():
    import bench

    n, p, ms = 200000, 50, 51.0
    entries = n * (n + 1) / 2
    for p_int in (0, 21):
        r = bench.lap_roofline(n, p, p_int, launches=2, ms=2 * ms, sm_count=152, sm_mhz=2000.0)
        assert r["bound"] == "alu" and r["unit"] == "Top/s"
        assert math.isclose(r["achieved"], entries * (2 * (p - p_int) + 2) / (ms * 1e-3) / 1e12, rel_tol=1e-12)
        assert math.isclose(r["peak"], 152 * 128 * 2000e6 / 1e12, rel_tol=1e-12)
        assert math.isclose(r["frac"], r["achieved"] / r["peak"], rel_tol=1e-12)
        q = r["integer_pipe"]
        assert math.isclose(q["achieved"], entries * p_int / (ms * 1e-3) / 1e12, rel_tol=1e-12, abs_tol=0.0)
        assert math.isclose(q["peak"], 152 * 64 * 2000e6 / 1e12, rel_tol=1e-12)
        assert math.isclose(r["lanes_frac"], r["frac"] + q["frac"], rel_tol=1e-12)
        assert r["traffic"] is not None
    assert bench.lap_roofline(1000, 20, 8, 1, 1.0, 152, 2000.0)["traffic"] is None


def test_split_follows_the_library_rule():
    import bench

    src = open(os.path.join(ROOT, "paper_2510_07929_gb300", "csrc", "abi.cu")).read()
    assert re.search(r"p >= 12 && std::ldexp\(\(double\)p, -G\) <= std::ldexp\(1\.0, -20\)", src)
    assert "std::lround(0.42 * (double)p)" in src and "if (G > 33) G = 33;" in src
    X = np.random.default_rng(0).uniform(-1, 1, (500, 50))
    assert bench.lap_int_features(X, 0.02) == 21
    assert bench.lap_int_features(X[:, :11], 0.1) == 0 and bench.lap_int_features(X[:, :12], 0.1) == 5
    X[0] += 300.0                       # the grid becomes too coarse
    assert bench.lap_int_features(X, 0.05) == 0
