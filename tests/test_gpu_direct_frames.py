"""Groups of cells in the direct cell kernel: a block's targets and the far
groups are taken relative to the centre of the targets' box.  Targets without a
position and targets far apart must leave their neighbours' field as it is."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import FIELD_TOL, guarded_rel_err, potential_err, pts4, to_dev
from paper_2110_09214_gb300 import inputs, obem

pytestmark = pytest.mark.gpu
NT = 32768 + 5


def _mesh(cells):
    m = inputs.parallel_plates(1e-3, 3e-4, int(np.ceil(np.sqrt(cells / 4))))
    mesh = inputs.Mesh(m.tri[:cells], m.kind[:cells], m.group[:cells], m.eps_minus[:cells], m.eps_plus[:cells],
                       m.group_voltage)
    cen = mesh.tri.mean(axis=1)
    return mesh, (1e-6 * (1.0 + 0.3 * np.sin(cen[:, 0] / 1e-4)) * np.where(cen[:, 2] > 1e-4, 1.0, -0.4)).astype(np.float32)


def _field(mesh, sigma, pts, capacity):
    ctx = obem.obem_create(capacity=capacity, dt=1e-12, flags=obem.OBEM_STEP_CELL_FIELD | obem.OBEM_STEP_CELL_GROUPS)
    try:
        obem.obem_mesh_load(ctx, mesh)
        out = torch.full((len(pts), 4), float("nan"), dtype=torch.float32, device="cuda")
        obem.obem_field_eval(ctx, to_dev(pts4(pts)), out, sigma=to_dev(sigma))
        torch.cuda.synchronize()
        return out.cpu().numpy()
    finally:
        obem.obem_destroy(ctx)


def _check(mesh, sigma, pts, got, idx):
    x, s = pts[idx].astype(np.float64), sigma.astype(np.float64)
    E, V = oracle.panel_field(mesh.tri, s, x)
    _, Vabs = oracle.panel_field(mesh.tri, np.abs(s), x)
    assert guarded_rel_err(got[idx, :3], E) <= FIELD_TOL
    assert potential_err(got[idx, 3], V, Vabs) <= FIELD_TOL


@pytest.mark.parametrize("capacity", [NT, 16])            # sorted targets, given order
def test_targets_without_a_position(capacity):
    mesh, sigma = _mesh(5001)
    rng = np.random.default_rng(3)
    pts = rng.uniform([0, 0, 4e-4], [1e-3, 1e-3, 2e-3], (NT, 3)).astype(np.float32)
    bad = np.arange(0, NT, 8 * 97)                         # the first of a block in the given order
    pts[bad, np.arange(len(bad)) % 3] = np.nan
    pts[bad[:5]] = np.nan
    got = _field(mesh, sigma, pts, capacity)
    rest = np.setdiff1d(np.arange(NT), bad)
    assert np.all(np.isfinite(got[rest]))
    _check(mesh, sigma, pts, got, rng.choice(rest, 512, replace=False))


@pytest.mark.parametrize("capacity", [NT, 16])
@pytest.mark.parametrize("extent", [1e-2, 10.0])
def test_targets_far_apart(extent, capacity):
    """Targets above the mesh, every other one up to `extent` to the side: a
    block of them cannot resolve a far group relative to its box."""
    mesh, sigma = _mesh(5001)
    rng = np.random.default_rng(4)
    pts = rng.uniform([0, 0, 4e-3], [1e-3, 1e-3, 8e-3], (NT, 3)).astype(np.float32)
    pts[::2, :2] += extent * rng.uniform(-1, 1, (len(pts[::2]), 2)).astype(np.float32)
    got = _field(mesh, sigma, pts, capacity)
    _check(mesh, sigma, pts, got, rng.choice(np.arange(1, NT, 2), 512, replace=False))
