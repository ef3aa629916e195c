"""Kernels whose lanes run over the cells or charges (sets of few targets):
block and warp remainders of the targets, cells and charges, and the sizes at
which the targets per block and the kernel change, against the oracle."""
import numpy as np
import pytest

import oracle
from gpu_util import FIELD_TOL, guarded_rel_err, potential_err, pts4, to_dev

pytestmark = pytest.mark.gpu


def _eval(ctx_capacity, mesh, sigma, pts, src=None, self_exclude=False):
    import torch
    from paper_2110_09214_gb300 import obem
    ctx = obem.obem_create(capacity=ctx_capacity, dt=1e-12)
    try:
        if mesh is not None:
            obem.obem_mesh_load(ctx, mesh)
        x = to_dev(pts4(pts))
        y = x if self_exclude else (to_dev(src) if src is not None else None)
        out = torch.full((len(pts), 4), float("nan"), dtype=torch.float32, device="cuda")
        obem.obem_field_eval(ctx, x, out, sources=y, self_exclude=self_exclude,
                             sigma=to_dev(sigma) if sigma is not None else None)
        torch.cuda.synchronize()
        return out.cpu().numpy()
    finally:
        obem.obem_destroy(ctx)


def _mesh(cells, rng):
    """The first `cells` triangles of two plates, the last ones a tenth the size (near and far tiers)."""
    from paper_2110_09214_gb300 import inputs
    m = inputs.parallel_plates(1e-3, 3e-4, max(2, int(np.ceil(np.sqrt(cells / 4)))))
    tri = m.tri[:cells].copy()
    small = tri[cells // 2:]
    small[:] = small.mean(axis=1, keepdims=True) + 0.1 * (small - small.mean(axis=1, keepdims=True))
    return inputs.Mesh(tri, m.kind[:cells], m.group[:cells], m.eps_minus[:cells], m.eps_plus[:cells],
                       m.group_voltage), rng.normal(0, 1e-6, cells).astype(np.float32)


@pytest.mark.parametrize("cells", [1, 33, 300])
@pytest.mark.parametrize("nt", [1, 2, 3, 8, 4095, 4097])
def test_cells(nt, cells):
    rng = np.random.default_rng(nt + 7 * cells)
    mesh, sigma = _mesh(cells, rng)
    pts = rng.uniform([0, 0, 0], [1e-3, 1e-3, 3e-4], (nt, 3)).astype(np.float32)
    got = _eval(max(nt, 16), mesh, sigma, pts)
    E, V = oracle.panel_field(mesh.tri, sigma.astype(np.float64), pts.astype(np.float64))
    _, Vabs = oracle.panel_field(mesh.tri, np.abs(sigma).astype(np.float64), pts.astype(np.float64))
    assert guarded_rel_err(got[:, :3], E) <= FIELD_TOL
    assert potential_err(got[:, 3], V, Vabs) <= FIELD_TOL


@pytest.mark.parametrize("nt,ns", [(1, 1), (2, 31), (9, 257), (4096, 33), (4095, 1000), (32769, 100)])
def test_charges_at_points(nt, ns):
    rng = np.random.default_rng(nt + 13 * ns)
    pts = rng.uniform(0, 1e-3, (nt, 3)).astype(np.float32)
    src = np.zeros((ns, 4), np.float32)
    src[:, :3] = rng.uniform(0, 1e-3, (ns, 3))
    src[:, 3] = 1.602176634e-19 * rng.choice([-1.0, 1.0], ns)
    got = _eval(16, None, None, pts, src=src)
    s64, p64 = src.astype(np.float64), pts.astype(np.float64)
    E, V = oracle.nbody_field(p64, s64, False)
    sabs = s64.copy()
    sabs[:, 3] = np.abs(sabs[:, 3])
    assert guarded_rel_err(got[:, :3], E) <= FIELD_TOL
    assert potential_err(got[:, 3], V, oracle.nbody_field(p64, sabs, False)[1]) <= FIELD_TOL


@pytest.mark.parametrize("n", [2, 257, 4097, 24576, 24577])
def test_charges_at_themselves(n):
    """Own charge left out, sets on both sides of the symmetric kernel's start."""
    rng = np.random.default_rng(n)
    q = np.zeros((n, 4), np.float32)
    q[:, :3] = rng.normal(0, 1e-4, (n, 3))
    q[:, 3] = 1.602176634e-19 * rng.choice([-1.0, 1.0], n)
    got = _eval(n, None, None, q, self_exclude=True)
    pick = rng.choice(n, min(n, 512), replace=False)
    s64 = q.astype(np.float64)
    E = np.empty((len(pick), 3))
    for k, i in enumerate(pick):
        d = s64[i, :3] - np.delete(s64, i, 0)[:, :3]
        w = 8.9875517923e9 * np.delete(s64, i, 0)[:, 3] / np.linalg.norm(d, axis=1) ** 3
        E[k] = (w[:, None] * d).sum(0)
    assert guarded_rel_err(got[pick, :3], E) <= FIELD_TOL
