"""The closed form in pairs of floats on cells so small that its products leave
binary32: those points are left to the FP64 form, the others agree with it."""
import numpy as np
import pytest

from test_closed_form_df_host import TOL, run  # noqa: F401  (the harness)


@pytest.mark.parametrize("h", [1e-13, 1e-12, 1e-11, 1e-10, 1e-9])
def test_small_cells(run, h):  # noqa: F811
    rng = np.random.default_rng(8)
    cases = []
    for _ in range(1500):
        v = rng.normal(0, h, (3, 3)) + rng.normal(0, 3 * h, 3)
        c, n = v.mean(0), np.cross(v[1] - v[0], v[2] - v[0])
        n /= np.linalg.norm(n)
        d = h * 10.0 ** rng.uniform(-2, 1)
        for p in (c + d * rng.normal(0, 1, 3), c + d * n, 0.5 * (v[0] + v[1]) - d * n):
            cases.append(np.concatenate([v.ravel(), p.astype(np.float32)]))
    out = run(cases)
    ok = out[:, 0] == 1
    assert np.all(np.isfinite(out[ok]))
    assert np.all(np.abs(out[ok, 2:5] - out[ok, 6:9]) <= TOL)
    assert np.all(np.abs(out[ok, 1] - out[ok, 5]) <= TOL * 10 * h)
    if h >= 1e-9:
        assert ok.mean() > 0.99
