"""The direct cell kernel's sorted targets and groups of cells in contexts that
can sort them: the sizes where the sort changes (one block up to 16,384
targets), where groups begin (32,768) and end, all targets in one bin or a
third, against the oracle and the given order."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import FIELD_TOL, guarded_rel_err, potential_err, pts4, to_dev
from paper_2110_09214_gb300 import inputs, obem

pytestmark = pytest.mark.gpu
GROUPS = obem.OBEM_STEP_CELL_GROUPS


def _mesh(cells):
    m = inputs.parallel_plates(1e-3, 3e-4, max(2, int(np.ceil(np.sqrt(cells / 4)))))
    mesh = inputs.Mesh(m.tri[:cells], m.kind[:cells], m.group[:cells], m.eps_minus[:cells], m.eps_plus[:cells],
                       m.group_voltage)
    cen = mesh.tri.mean(axis=1)
    return mesh, (1e-6 * (1.0 + 0.3 * np.sin(cen[:, 0] / 1e-4)) *
                  np.where(mesh.group % 2 == 0, 1.0, -1.0)).astype(np.float32)


def _field(mesh, sigma, pts, capacity, flags):
    ctx = obem.obem_create(capacity=capacity, dt=1e-12, flags=obem.OBEM_STEP_CELL_FIELD | flags)
    try:
        obem.obem_mesh_load(ctx, mesh)
        out = torch.full((len(pts), 4), float("nan"), dtype=torch.float32, device="cuda")
        obem.obem_field_eval(ctx, to_dev(pts4(pts)), out, sigma=to_dev(sigma))
        torch.cuda.synchronize()
        return out.cpu().numpy()
    finally:
        obem.obem_destroy(ctx)


@pytest.mark.parametrize("one_bin", ["third", "all", "none"])
@pytest.mark.parametrize("nt,cells,flags", [
    (4096, 33, 0), (5000, 1001, 0), (16383, 33, 0), (16384, 33, 0), (16385, 33, 0), (32767, 1001, GROUPS),
    (32768, 31, GROUPS), (32768, 33, GROUPS), (32775, 5001, GROUPS)])
def test_sorted_targets(nt, cells, flags, one_bin):
    mesh, sigma = _mesh(cells)
    rng = np.random.default_rng(nt + cells)
    pts = rng.uniform([0, 0, 0], [1e-3, 1e-3, 3e-4], (nt, 3)).astype(np.float32)
    k = {"third": nt // 3, "all": nt, "none": 0}[one_bin]
    pts[:k] = np.float32([4.4e-4, 6.1e-4, 1.3e-4]) + (1e-7 * rng.standard_normal((k, 3))).astype(np.float32)
    got = _field(mesh, sigma, pts, nt, flags)
    assert np.all(np.isfinite(got))
    idx = np.unique(np.concatenate([[0, nt // 3, nt - 1], rng.choice(nt, 509, replace=False)]))
    x, s = pts[idx].astype(np.float64), sigma.astype(np.float64)
    E, V = oracle.panel_field(mesh.tri, s, x)
    _, Vabs = oracle.panel_field(mesh.tri, np.abs(s), x)
    assert guarded_rel_err(got[idx, :3], E) <= FIELD_TOL
    assert potential_err(got[idx, 3], V, Vabs) <= FIELD_TOL
    # every target of the set against the given order (a context of 16): the same
    # field to the two orders' rounding, so no target is left out or taken twice
    other = _field(mesh, sigma, pts, 16, flags)
    assert guarded_rel_err(got[:, :3], other[:, :3]) <= 2 * FIELD_TOL
