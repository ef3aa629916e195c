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
