"""The closed form of the cell integrals in pairs of floats against the FP64 form,
both run on the CPU through a native harness: points from a thousandth of a
cell size to a few sizes away, above the cell, beside and beyond its edges; and
the points that it must leave to the FP64 form."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
# Vertices and points lie within ~40 cell sizes of the origin and 1e-4 sizes and
# more apart; a pair holds a coordinate to 2^-48 of its value, so a distance to
# 40 / 1e-4 x 2^-48 = 1.4e-9 of its own at worst, which three logarithms and the
# angle turn into as many absolute 1e-9s.  A binary32 ulp of F is 1e-7 and more.
TOL = 1e-8


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    nvcc = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    nvcc = nvcc if os.path.exists(nvcc) else shutil.which("nvcc")
    if not nvcc:
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("cfdf")
    exe = str(d / "harness")
    r = subprocess.run([nvcc, "-O2", "-std=c++17", "-Xcompiler", "-ffp-contract=off", "-I", os.path.join(ROOT, "include"),
                        "-o", exe, os.path.join(HERE, "native", "closed_form_df_host.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def f(cases):
        cases = np.ascontiguousarray(cases, np.float64)
        (d / "in").write_bytes(struct.pack("i", len(cases)) + cases.tobytes())
        r = subprocess.run([exe, str(d / "in"), str(d / "out")], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return np.frombuffer((d / "out").read_bytes(), np.float64).reshape(len(cases), 9)
    return f


@pytest.mark.parametrize("h", [1e-7, 1e-4, 1.0])
def test_pairs_of_floats(run, h):
    rng = np.random.default_rng(5)
    cases = []
    for _ in range(1500):
        v = rng.normal(0, h, (3, 3)) + rng.normal(0, 10 * h, 3)
        c, n = v.mean(0), np.cross(v[1] - v[0], v[2] - v[0])
        n /= np.linalg.norm(n)
        e, w = (v[1] - v[0]) / np.linalg.norm(v[1] - v[0]), rng.dirichlet([1, 1, 1])
        d = h * 10.0 ** rng.uniform(-3, 0.5)
        for p in (c + d * rng.normal(0, 1, 3), w @ v + d * n, w @ v - d * n, v[0] - 0.7 * d * e + 0.1 * d * n,
                  0.5 * (v[0] + v[1]) + d * np.cross(e, n)):
            cases.append(np.concatenate([v.ravel(), p.astype(np.float32)]))
    out = run(cases)
    assert np.all(out[:, 0] == 1)
    assert np.all(np.abs(out[:, 2:5] - out[:, 6:9]) <= TOL)
    assert np.all(np.abs(out[:, 1] - out[:, 5]) <= TOL * 10 * h)
    # what leaves the kernels: the same binary32 number but for one in a thousand
    same = out[:, 1:5].astype(np.float32) == out[:, 5:9].astype(np.float32)
    assert same.mean() > 0.999


def test_left_to_fp64(run):
    v = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0]], np.float64)
    pts = {(0.5, 0.0, 0.0): 0, (0.0, 0.0, 0.0): 0, (0.5, 0.0, 1e-9): 0, (0.25, 0.25, 1e-14): 0,
           (0.25, 0.25, 0.0): 1, (2.0, 2.0, 0.0): 1, (-1.0, 0.0, 0.0): 1, (0.25, 0.25, 1e-6): 1, (0.25, 0.25, -1e-3): 1, (0.5, -1e-4, 0.0): 1}
    out = run([np.concatenate([v.ravel(), np.float32(p)]) for p in pts])
    assert out[:, 0].tolist() == list(pts.values())
    ok = out[:, 0] == 1
    assert np.all(np.abs(out[ok, 1:5] - out[ok, 5:9]) <= TOL)
