"""Fields on both sides of the sizes where the direct kernels hand over to the
block kernels, against the oracle."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import FIELD_TOL, guarded_rel_err, potential_err, pts4, to_dev
from paper_2110_09214_gb300 import obem

pytestmark = pytest.mark.gpu
E = 1.602176634e-19


@pytest.mark.parametrize("nt,ns", [(12_288, 1), (12_288, 256), (12_289, 1), (12_289, 256), (12_289, 257), (32_769, 257)])
def test_few_charges_at_points(nt, ns):
    rng = np.random.default_rng(nt + ns)
    pts = rng.uniform(0, 1e-3, (nt, 3)).astype(np.float32)
    src = np.column_stack([rng.uniform(0, 1e-3, (ns, 3)), E * rng.choice([-1.0, 1.0], ns)]).astype(np.float32)
    ctx = obem.obem_create(capacity=16, dt=1e-12)
    try:
        out = torch.full((nt, 4), float("nan"), dtype=torch.float32, device="cuda")
        obem.obem_field_eval(ctx, to_dev(pts4(pts)), out, sources=to_dev(src))
        torch.cuda.synchronize()
        got = out.cpu().numpy()
    finally:
        obem.obem_destroy(ctx)
    s64, p64 = src.astype(np.float64), pts.astype(np.float64)
    ref, V = oracle.nbody_field(p64, s64, False)
    s64[:, 3] = np.abs(s64[:, 3])
    assert guarded_rel_err(got[:, :3], ref) <= FIELD_TOL
    assert potential_err(got[:, 3], V, oracle.nbody_field(p64, s64, False)[1]) <= FIELD_TOL


@pytest.fixture(scope="module")
def plates():
    from paper_2110_09214_gb300 import inputs
    mesh = inputs.parallel_plates(1e-2, 1e-3, 36)
    cen = mesh.tri.mean(axis=1)
    return mesh, (1e-6 * (1.0 + 0.3 * np.sin(cen[:, 0] / 1e-3)) * np.where(cen[:, 2] > 5e-4, 1.0, -1.0)).astype(np.float32)


def _points(kind, n, rng):
    if kind == "cloud":
        return np.array([5e-3, 5e-3, 4e-5]) + rng.normal(0, 1e-5, (n, 3))
    p = rng.uniform([0, 0, 0], [1e-2, 1e-2, 1e-3], (n, 3))
    if kind == "both":                                   # full blocks beside nearly empty ones
        p[: 3 * n // 4] = np.array([2e-3, 3e-3, 5e-4]) + rng.normal(0, 2e-5, (3 * n // 4, 3))
    return p


@pytest.mark.parametrize("flags", [obem.OBEM_STEP_CELL_FIELD, obem.OBEM_STEP_CELL_FIELD | obem.OBEM_STEP_CELL_GROUPS])
@pytest.mark.parametrize("kind", ["cloud", "spread", "both"])
@pytest.mark.parametrize("nt", [196_608, 196_609, 262_147, 458_753])
def test_many_targets_either_kernel(plates, nt, kind, flags):
    """Above 196,608 targets the block list says whether the block kernels or
    the direct one evaluate the cells: every target gets its field once."""
    mesh, sigma = plates
    rng = np.random.default_rng(nt)
    pts = _points(kind, nt, rng).astype(np.float32)
    ctx = obem.obem_create(capacity=nt, dt=1e-12, flags=flags)
    try:
        obem.obem_mesh_load(ctx, mesh)
        out = torch.full((nt, 4), float("nan"), dtype=torch.float32, device="cuda")
        obem.obem_field_eval(ctx, to_dev(pts4(pts)), out, sigma=to_dev(sigma))
        obem.obem_field_eval(ctx, to_dev(pts4(pts)), out, sigma=to_dev(sigma))       # on top of the first's results
        torch.cuda.synchronize()
        got = out.cpu().numpy()
    finally:
        obem.obem_destroy(ctx)
    assert np.all(np.isfinite(got))
    idx = np.unique(np.concatenate([[0, nt // 2, nt - 1], rng.choice(nt, 256, replace=False)]))
    x, s = pts[idx].astype(np.float64), sigma.astype(np.float64)
    ref, V = oracle.panel_field(mesh.tri, s, x)
    _, Vabs = oracle.panel_field(mesh.tri, np.abs(s), x)
    assert guarded_rel_err(got[idx, :3], ref) <= FIELD_TOL
    assert potential_err(got[idx, 3], V, Vabs) <= FIELD_TOL


@pytest.mark.parametrize("flags", [obem.OBEM_STEP_CELL_FIELD, obem.OBEM_STEP_CELL_FIELD | obem.OBEM_STEP_CELL_GROUPS])
@pytest.mark.parametrize("kind", ["cloud", "spread", "outlier"])
@pytest.mark.parametrize("nt", [65_535, 65_536, 131_073, 262_147])
def test_many_targets_in_the_given_order(plates, nt, kind, flags):
    """More targets than the context can sort: the near cells of their blocks
    say which kernels take them (outlier: a cloud with a few far points, whose
    blocks are near many cells)."""
    mesh, sigma = plates
    rng = np.random.default_rng(nt)
    pts = _points("spread" if kind == "spread" else "cloud", nt, rng).astype(np.float32)
    if kind == "outlier":
        pts[[7, nt // 3, nt - 1]] = [[1e-3, 9e-3, 9e-4], [9e-3, 1e-3, 1e-4], [5e-3, 5e-3, 5e-2]]
    ctx = obem.obem_create(capacity=16, dt=1e-12, flags=flags)
    try:
        obem.obem_mesh_load(ctx, mesh)
        out = torch.full((nt, 4), float("nan"), dtype=torch.float32, device="cuda")
        obem.obem_field_eval(ctx, to_dev(pts4(pts)), out, sigma=to_dev(sigma))
        obem.obem_field_eval(ctx, to_dev(pts4(pts)), out, sigma=to_dev(sigma))
        torch.cuda.synchronize()
        got = out.cpu().numpy()
    finally:
        obem.obem_destroy(ctx)
    assert np.all(np.isfinite(got))
    idx = np.unique(np.concatenate([[0, 7, nt // 3, nt - 1], rng.choice(nt, 256, replace=False)]))
    x, s = pts[idx].astype(np.float64), sigma.astype(np.float64)
    ref, V = oracle.panel_field(mesh.tri, s, x)
    _, Vabs = oracle.panel_field(mesh.tri, np.abs(s), x)
    assert guarded_rel_err(got[idx, :3], ref) <= FIELD_TOL
    assert potential_err(got[idx, 3], V, Vabs) <= FIELD_TOL


def test_unsorted_calls_on_two_streams(plates):
    """A cloud and a spread-out set alternating on two streams of one context:
    each call has its own decision."""
    mesh, sigma = plates
    rng = np.random.default_rng(12)
    nt = 65_536
    sets = [_points(kind, nt, rng).astype(np.float32) for kind in ("cloud", "spread")]
    sg = to_dev(sigma)
    x = [to_dev(pts4(p)) for p in sets]
    ctx = obem.obem_create(capacity=16, dt=1e-12, flags=obem.OBEM_STEP_CELL_FIELD)
    try:
        obem.obem_mesh_load(ctx, mesh)
        want = []
        for k in range(2):
            o = torch.full((nt, 4), float("nan"), dtype=torch.float32, device="cuda")
            obem.obem_field_eval(ctx, x[k], o, sigma=sg)
            torch.cuda.synchronize()
            want.append(o)
        streams = [torch.cuda.Stream(), torch.cuda.Stream()]
        out = [[torch.full((nt, 4), float("nan"), dtype=torch.float32, device="cuda") for _ in range(12)] for _ in range(2)]
        torch.cuda.synchronize()
        for r in range(12):
            for k in range(2):
                obem.obem_field_eval(ctx, x[k], out[k][r], sigma=sg, stream=streams[k])
        torch.cuda.synchronize()
        for k in range(2):
            for o in out[k]:
                assert torch.equal(o, want[k])
    finally:
        obem.obem_destroy(ctx)


def test_live_count_decides(plates):
    """A state of 300,000 slots holding 2000 and 250,000 electrons at rest: the
    cells' field of either kernel moves them (v = (q/m) E dt)."""
    from paper_2110_09214_gb300 import inputs
    mesh, sigma = plates
    cap, dt = 300_000, 1e-15
    ctx = obem.obem_create(capacity=cap, dt=dt, z_lo=-1.0, z_hi=1.0, beta=-1.0, flags=obem.OBEM_STEP_CELL_FIELD)
    try:
        obem.obem_gas_load(ctx, inputs.maxwell_gas(0.0, 0.0))
        obem.obem_mesh_load(ctx, mesh)
        obem.obem_bem_assemble(ctx, obem.OBEM_LU_BF16)
        sig = torch.empty(mesh.n, dtype=torch.float32, device="cuda")
        obem.obem_bem_solve(ctx, np.array([0.0, 500.0]), sig)
        s = sig.cpu().numpy().astype(np.float64)
        for n in (2000, 250_000):
            rng = np.random.default_rng(n)
            pos = _points("cloud", n, rng)
            st = obem.DeviceState(cap)
            st.upload(inputs.make_charges(pos, np.zeros((n, 3)), np.zeros(n, np.uint8)))
            stats = obem.new_stats()
            obem.obem_step(ctx, st, 0, stats)
            out, _ = st.download()
            assert out.n == n and obem.read_stats(stats)["status"] == 0
            qm = -1.602176634e-19 / 9.1093837015e-31
            got = out.vel[:, :3].astype(np.float64) / (float(np.float32(qm)) * float(np.float32(dt)))
            idx = rng.choice(n, 256, replace=False)
            ref, _ = oracle.panel_field(mesh.tri, s, pos[idx].astype(np.float32).astype(np.float64))
            assert guarded_rel_err(got[idx], ref) <= FIELD_TOL
    finally:
        obem.obem_destroy(ctx)
