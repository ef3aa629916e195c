"""The FP64 closed form of the cell integrals as the GPU kernels have it, run on
the CPU through a native harness, against the same expressions with the C
library's square root, logarithm and arc tangent (and, coarsely, against the
oracle): points from a thousandth of a cell size away to many sizes, in the
cell's plane, beside and beyond its edges; and those functions against
numpy's over 60 decades, zeros among the arguments."""
import os
import shutil
import struct
import subprocess

import numpy as np
import pytest

import oracle

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
# The functions are accurate to ~1e-15; a logarithm is at most ~15 and a solid
# angle 2 pi here, so F, the sum of three logarithms and the angle, may differ by
# 3 x 15e-15 + 6e-15, and phi by as much times the distances that multiply them;
# the square roots' errors enter the logarithms' arguments (1e-15 each).
TOL = 1e-13


def _nvcc():
    p = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "bin", "nvcc")
    return p if os.path.exists(p) else shutil.which("nvcc")


@pytest.fixture(scope="module")
def harness(tmp_path_factory):
    if not _nvcc():
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("cf")
    exe = str(d / "harness")
    r = subprocess.run([_nvcc(), "-O2", "-std=c++17", "-I", os.path.join(ROOT, "include"), "-o", exe,
                        os.path.join(HERE, "native", "closed_form_host.cu")], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr

    def run(cases):
        cases = np.ascontiguousarray(cases, np.float64)
        (d / "in").write_bytes(struct.pack("i", len(cases)) + cases.tobytes())
        r = subprocess.run([exe, str(d / "in"), str(d / "out")], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr
        return np.frombuffer((d / "out").read_bytes(), np.float64).reshape(len(cases), 16)
    return run


@pytest.mark.parametrize("h", [1e-6, 1e-3, 1.0])
def test_integrals(harness, h):
    rng = np.random.default_rng(3)
    cases = []
    for _ in range(400):
        v = rng.normal(0, h, (3, 3)) + rng.normal(0, 10 * h, 3)
        c, n = v.mean(0), np.cross(v[1] - v[0], v[2] - v[0])
        n /= np.linalg.norm(n)
        e, w = v[1] - v[0], rng.dirichlet([1, 1, 1])
        d = h * 10.0 ** rng.uniform(-3, 2)
        cases += [np.concatenate([v.ravel(), p]) for p in (
            c + d * rng.normal(0, 1, 3),                # anywhere
            w @ v + d * n,                              # above the cell
            v[0] - 0.7 * d * e / np.linalg.norm(e) + 0.1 * d * n,      # beyond a vertex, beside an edge's line
            0.5 * (v[0] + v[1]) + d * np.cross(e, n) / np.linalg.norm(e))]     # beside an edge
    out = harness(cases)
    assert np.all(np.abs(out[:, 4] - out[:, 8]) <= TOL * out[:, 12])
    assert np.all(np.abs(out[:, 5:8] - out[:, 9:12]) <= TOL)
    for k in range(0, len(cases), 7):
        phi, F = oracle.tri_integrals(cases[k][:9], cases[k][9:])
        for o in (out[k, :4], out[k, 4:8]):
            assert abs(o[0] - phi) <= 1e-9 * out[k, 12] and np.linalg.norm(o[1:] - F) <= 1e-9


def test_in_plane_and_on_the_edge(harness):
    v = np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0]], np.float64)
    out = harness([np.concatenate([v.ravel(), p]) for p in ([0.25, 0.25, 0], [2, 2, 0], [0.5, 0, 0], [0, 0, 0])])
    with np.errstate(invalid="ignore"):
        same = np.abs(out[:, 4:8] - out[:, 8:12]) <= TOL
    assert np.all(same | ~np.isfinite(out[:, 8:12])) and np.all(np.isfinite(out[:, 4:8]) == np.isfinite(out[:, 8:12]))


def test_functions(harness):
    rng = np.random.default_rng(4)
    n = 4000
    x = np.concatenate([10.0 ** rng.uniform(-30, 30, (n, 5)), rng.uniform(0.5, 2, (n, 5)),
                        1 + 10.0 ** rng.uniform(-15, -1, (n, 5)), 10.0 ** rng.uniform(-300, 300, (n, 5))])
    x[:, 3:5] *= rng.choice([-1.0, 1.0], (len(x), 2))
    x = np.concatenate([x, [[0, 1, 2, 0, 1], [1, 2, 2, 0, -1], [4, 1e-320, 3, 1, 0], [2, 3, 3, -1, 0]]])
    cases = np.zeros((len(x), 12))
    cases[:, :9] = [0, 0, 0, 1, 0, 0, 0, 1, 0]
    cases[:, 9:] = 0.3
    cases[:, :5] = x
    out = harness(cases)[:, 13:]
    assert np.all(np.abs(out[:, 0] - np.sqrt(x[:, 0])) <= 5e-14 * np.sqrt(x[:, 0]))
    a, b = x[:, 1].astype(np.longdouble), x[:, 2].astype(np.longdouble)
    near = np.abs(a / b - 1) < 0.5
    ref = np.where(near, np.log1p(np.where(near, (a - b) / b, 0)), np.log(a) - np.log(b)).astype(np.float64)
    assert np.all(np.abs(out[:, 1] - ref) <= 5e-14 * np.abs(ref))
    ref = np.arctan2(x[:, 3], x[:, 4])
    assert np.all(np.abs(out[:, 2] - ref) <= 5e-14 * np.abs(ref))
