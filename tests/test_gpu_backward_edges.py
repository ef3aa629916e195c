"""Gradients of the field where charges or targets have no position, and at the
sizes where the kernels change, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import FIELD_TOL, grad_abs_scales, grad_err, pts4, to_dev
from paper_2110_09214_gb300 import obem

pytestmark = pytest.mark.gpu
E = 1.602176634e-19


def _inputs(nt, ns, seed):
    rng = np.random.default_rng(seed)
    tgt = rng.uniform(-2e-4, 1.2e-3, (nt, 3)).astype(np.float32)
    src = np.column_stack([rng.uniform(0, 1e-3, (ns, 3)), rng.choice([-E, E], ns)]).astype(np.float32)
    g = (rng.normal(0, 1.0, (nt, 4)) * [1, 1, 1, 1e3]).astype(np.float32)
    return tgt, src, g


def _backward(tgt, g, src, mesh=None, sigma=None):
    ctx = obem.obem_create(capacity=16, dt=1e-12)
    try:
        if mesh is not None:
            obem.obem_mesh_load(ctx, mesh)
        dt = torch.full((len(tgt), 4), float("nan"), device="cuda")
        ds = torch.full((len(src), 4), float("nan"), device="cuda") if src is not None else None
        obem.obem_field_eval_backward(ctx, to_dev(pts4(tgt)), to_dev(g), sources=None if src is None else to_dev(src),
                                      sigma=None if sigma is None else to_dev(sigma), dL_dtargets=dt, dL_dsources=ds)
        torch.cuda.synchronize()
        return dt.cpu().numpy().astype(np.float64), None if ds is None else ds.cpu().numpy().astype(np.float64)
    finally:
        obem.obem_destroy(ctx)


def _check(tgt, g, src, dt, ds):
    _, rt, rs = oracle.field_backward(None, None, tgt.astype(np.float64), src.astype(np.float64), False,
                                      g.astype(np.float64))
    _, at, ap, aq = grad_abs_scales(tgt, g, src)
    assert grad_err(dt[:, :3], rt, at) <= FIELD_TOL
    assert grad_err(ds[:, :3], rs[:, :3], ap) <= FIELD_TOL
    assert grad_err(ds[:, 3], rs[:, 3], aq) <= FIELD_TOL


@pytest.mark.parametrize("nt,ns", [(101, 70), (300, 1500), (9, 50_000)])
def test_charges_and_targets_without_a_position(nt, ns):
    """They give no term and have no gradient, also where the upstream gradient
    is NaN; the others' gradients are those without them."""
    tgt, src, g = _inputs(nt, ns, nt + ns)
    bt, bs = np.array([0, 3, 4, nt - 1]), np.array([1, 2, 33, ns - 1])
    tgt[bt, np.arange(4) % 3] = np.nan
    src[bs, np.arange(4) % 3] = np.nan
    tgt[4], src[33, :3] = np.nan, np.nan
    g[3] = np.nan
    dt, ds = _backward(tgt, g, src)
    assert np.all(dt[bt] == 0.0) and np.all(ds[bs] == 0.0)
    kt, ks = np.setdiff1d(np.arange(nt), bt), np.setdiff1d(np.arange(ns), bs)
    _check(tgt[kt], g[kt], src[ks], dt[kt], ds[ks])


@pytest.mark.parametrize("nt,ns", [(1, 31), (17, 255), (1, 65_536), (128, 65_535), (128, 65_537), (129, 65_600),
                                   (2, 262_143), (129, 262_145)])
def test_sources_split_or_not(nt, ns):
    """dL/dy and dL/dq on both sides of the sizes where the targets are no
    longer split over the warps, blocks of sources partly filled."""
    tgt, src, g = _inputs(nt, ns, nt + ns)
    dt, ds = _backward(tgt, g, src)
    pick = np.unique(np.concatenate([[0, ns - 1], np.random.default_rng(5).choice(ns, min(ns, 2000), replace=False)]))
    _, _, rs = oracle.field_backward(None, None, tgt.astype(np.float64), src[pick].astype(np.float64), False,
                                     g.astype(np.float64))
    _, _, ap, aq = grad_abs_scales(tgt, g, src[pick])
    assert np.all(np.isfinite(ds))
    assert grad_err(ds[pick, :3], rs[:, :3], ap) <= FIELD_TOL
    assert grad_err(ds[pick, 3], rs[:, 3], aq) <= FIELD_TOL


@pytest.mark.parametrize("nt", [1, 5, 70_001])
def test_no_charges_and_no_cells(nt):
    tgt, _, g = _inputs(nt, 1, nt)
    dt, _ = _backward(tgt, g, None)
    assert np.all(dt == 0.0)


def _near_mesh(cells, rng):
    """Triangles of about 1 mm whose centroids lie within 0.1 mm: every target
    near is within 1.5 h of all of them."""
    from paper_2110_09214_gb300 import inputs
    tri = rng.normal(0, 5e-4, (cells, 3, 3))
    tri += rng.normal(0, 3e-5, (cells, 1, 3)) - tri.mean(axis=1, keepdims=True)
    z = np.zeros(cells, np.int32)
    return inputs.Mesh(tri, z, z, np.ones(cells), np.ones(cells), np.array([1.0])), \
        rng.normal(0, 1e-6, cells).astype(np.float32)


@pytest.mark.parametrize("nt,cells", [(1, 1), (5, 4), (4, 32), (9, 33), (130, 100), (3, 700), (6, 1300)])
def test_targets_near_every_cell(nt, cells):
    """dL/dx where all pairs take the closed form: meshes of a warp's share and
    less, and queues that are emptied before the end."""
    rng = np.random.default_rng(nt + cells)
    mesh, sigma = _near_mesh(cells, rng)
    tgt = rng.normal(0, 2e-5, (nt, 3)).astype(np.float32)
    g = (rng.normal(0, 1.0, (nt, 4)) * [1, 1, 1, 1e3]).astype(np.float32)
    dt, _ = _backward(tgt, g, None, mesh, sigma)
    _, rt, _ = oracle.field_backward(mesh.tri, sigma.astype(np.float64), tgt.astype(np.float64), None, False,
                                     g.astype(np.float64))
    _, at, _, _ = grad_abs_scales(tgt, g, None, mesh.tri, sigma)
    assert np.all(dt[:, 3] == 0.0)
    assert grad_err(dt[:, :3], rt, at) <= FIELD_TOL
