"""Batches too large for the direct cell kernel: the block kernels of chambers,
at the block sizes, against the oracle chamber by chamber."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import FIELD_TOL, guarded_rel_err
from paper_2110_09214_gb300 import inputs, obem

pytestmark = pytest.mark.gpu
SOFT = 1e-9


@pytest.mark.parametrize("caps", [[40_960, 30_720, 26_624], [60_000, 1024, 50_000]])      # 98,304 slots: direct; more: blocks
def test_cells_of_large_batches(caps):
    rng = np.random.default_rng(sum(caps))
    gaps, sizes = [6e-4, 1e-3, 2e-3], [900, 1, 2100]
    ctx = obem.obem_create(capacity=16, dt=1e-12, softening=SOFT, beta=1e-13,
                           flags=obem.OBEM_STEP_SPACE_CHARGE | obem.OBEM_STEP_CELL_FIELD)
    b = None
    try:
        obem.obem_gas_load(ctx, inputs.argon_like_gas())
        chs, cells = [], []
        for k, (gap, n) in enumerate(zip(gaps, sizes)):
            mesh = inputs.parallel_plates(1e-2, gap, 3 + k, 0.0, 1e6 * gap)
            ch = inputs.avalanche_snapshot(rng, n, gap=gap)
            ch.pos_q[:, 2] = np.clip(ch.pos_q[:, 2], 0.05 * gap, 0.95 * gap)
            chs.append(ch)
            cells.append((mesh, oracle.bem_solve(mesh).astype(np.float32)))
        b = obem.Batch(ctx, caps, [0.0] * 3, gaps, [1, 2, 3])
        assert (int(b.seg_off[-1]) > 98_304) == (caps[1] == 1024)
        for k, (mesh, sigma) in enumerate(cells):
            b.cells(k, mesh.tri, sigma)
        st = b.state()
        st.upload(chs)
        fields = {}
        for cut in (64, 128, 512):
            b.set_block(cut)
            out = torch.full((st.capacity, 4), float("nan"), device="cuda")
            b.field_eval(st, out)
            torch.cuda.synchronize()
            fields[cut] = out.cpu().numpy().astype(np.float64)
        r = b.autotune(st, reps=2)
        assert r["cells_per_block"] in (128, 256, 512) and r["ms"] > 0
    finally:
        if b is not None:
            b.destroy()
        obem.obem_destroy(ctx)
    for k, (ch, (mesh, sigma)) in enumerate(zip(chs, cells)):
        o, pts = int(b.seg_off[k]), ch.pos_q[:, :3].astype(np.float64)
        ref = oracle.panel_field(mesh.tri, sigma.astype(np.float64), pts)[0]
        ref = ref + oracle.nbody_field(pts, ch.pos_q.astype(np.float64), True, SOFT)[0]
        for cut, got in fields.items():
            assert np.all(np.isfinite(got[o:o + ch.n])), (k, cut)
            assert guarded_rel_err(got[o:o + ch.n, :3], ref) <= FIELD_TOL, (k, cut)
