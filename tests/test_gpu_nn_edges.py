"""Approximate N-body field where pairs have no distance or charges no position,
against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2110_09214_gb300 import obem
from gpu_util import FIELD_TOL, guarded_rel_err, to_dev

pytestmark = pytest.mark.gpu
E = 1.602176634e-19


def _clouds(n, seed, weight):
    rng = np.random.default_rng(seed)
    p = rng.normal(0, 2e-5, (n, 3))
    return np.column_stack([p, weight * E * rng.choice([-1.0, 1.0], n)]).astype(np.float32)


def _gpu_nn(src, grid, soft):
    ctx = obem.obem_create(capacity=max(len(src), 16), dt=1e-12)
    try:
        out = torch.full((len(src), 4), float("nan"), device="cuda")
        obem.obem_nbody_nn_eval(ctx, to_dev(src), out, grid, soft)
        torch.cuda.synchronize()
        return out.cpu().numpy().astype(np.float64)
    finally:
        obem.obem_destroy(ctx)


@pytest.mark.parametrize("soft", [0.0, 1e-9])
@pytest.mark.parametrize("weight", [1.0, 200.0, 1e3, 1e6])
@pytest.mark.parametrize("n,grid", [(64, 4), (300, 1), (3000, 8)])
def test_nn_charges_at_one_point(n, grid, weight, soft):
    """Macro-charges at the same point (pairs of either sign, a stack of more
    than a warp's lanes): such a pair gives no term."""
    src = _clouds(n, n + grid, weight)
    src[10, :3] = src[11, :3]
    src[10, 3], src[11, 3] = src[11, 3], -src[11, 3]
    src[20:20 + 40, :3] = src[20, :3]
    src[n - 1, :3] = src[0, :3]
    src[n - 1, 3] = src[0, 3]
    got = _gpu_nn(src, grid, soft)
    assert np.all(np.isfinite(got))
    assert guarded_rel_err(got[:, :3], oracle.nbody_nn(src.astype(np.float64), grid, soft)) <= FIELD_TOL


@pytest.mark.parametrize("grid", [1, 4, 8])
def test_nn_charges_without_a_position(grid):
    """A charge with a NaN coordinate gives no term and gets none; the others
    see each other as without it."""
    src = _clouds(3000, 77, 1.0)
    bad = np.array([0, 7, 8, 9, 1500, 2999])
    src[bad, np.array([0, 1, 2, 0, 1, 2])] = np.nan
    src[8, :3] = np.nan
    got = _gpu_nn(src, grid, 1e-9)
    rest = np.setdiff1d(np.arange(3000), bad)
    assert np.all(got[bad] == 0.0)
    assert guarded_rel_err(got[rest, :3], oracle.nbody_nn(src[rest].astype(np.float64), grid, 1e-9)) <= FIELD_TOL
