"""The fit of the cell groups kept for the context's own densities, at sizes whose
step takes the groups: in the direct kernel and in the block kernels."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import FIELD_TOL, guarded_rel_err
from paper_2110_09214_gb300 import inputs, obem

pytestmark = pytest.mark.gpu
QM = float(np.float32(-1.602176634e-19 / 9.1093837015e-31))


@pytest.fixture(scope="module")
def gem():
    mesh, gas, ch, trk, g = inputs.config_gem(seed=4, n=60_000, target_panels=20_000)
    return mesh, ch, g


def _fields(mesh, g, el, flags, scales):
    """The cells' field at electrons at rest, read back from a step's
    velocities, after a solve for every scale of the voltages."""
    n, dt = len(el), 1e-15
    ctx = obem.obem_create(capacity=n + 64, dt=dt, z_lo=g.z_anode - 1e-3, z_hi=g.z_drift + 1e-3, beta=-1.0,
                           flags=obem.OBEM_STEP_CELL_FIELD | flags)
    try:
        obem.obem_gas_load(ctx, inputs.maxwell_gas(0.0, 0.0))
        obem.obem_mesh_load(ctx, mesh)
        obem.obem_bem_assemble(ctx, obem.OBEM_LU_BF16)
        st, stats = obem.DeviceState(n + 64), obem.new_stats()
        sig = torch.empty(mesh.n, dtype=torch.float32, device="cuda")
        out = []
        for scale in scales:
            gv = np.asarray(mesh.group_voltage, np.float64) * scale
            gv[0] += 37.0 * (scale != 1.0)
            obem.obem_bem_solve(ctx, gv, sig)
            st.upload(inputs.make_charges(el, np.zeros((n, 3)), np.zeros(n, np.uint8)))
            obem.obem_step(ctx, st, 0, stats)
            torch.cuda.synchronize()
            assert obem.read_stats(stats)["status"] == 0
            res, _ = st.download()
            assert res.n == n
            out.append((res.vel[:, :3].copy(), sig.cpu().numpy().astype(np.float64)))
        return out, QM * float(np.float32(dt))
    finally:
        obem.obem_destroy(ctx)


@pytest.mark.parametrize("n", [33_000, 460_000])
def test_kept_fit_follows_a_new_solve(gem, n):
    mesh, ch, g = gem
    rng = np.random.default_rng(n)
    base = ch.pos_q[rng.integers(0, ch.n, n), :3].astype(np.float64)
    el = (base + rng.normal(0, 1e-7, (n, 3))).astype(np.float32).astype(np.float64)
    idx = np.sort(rng.choice(n, 512, replace=False))
    grouped, f = _fields(mesh, g, el, obem.OBEM_STEP_CELL_GROUPS, (1.0, 0.6))
    plain, _ = _fields(mesh, g, el, 0, (1.0,))
    # the groups were used: their far field differs in the last bits
    assert (grouped[0][0] != plain[0][0]).any(axis=1).mean() > 0.25
    for vel, sigma in grouped:
        ref, _ = oracle.panel_field(mesh.tri, sigma, el[idx])
        assert guarded_rel_err(vel[idx].astype(np.float64) / f, ref) <= FIELD_TOL
