"""Kernels chosen by the size of a context or a batch, on both sides of every
line: the tracking step's chunks (8, 32, 128 and 256 charges per warp, moments of
256 and 1024 per block) give the same bits whatever the capacity, and the batched
all-pairs sum in units of 1, 4 and 16 tile pairs the oracle's field."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import FIELD_TOL, guarded_rel_err
from paper_2110_09214_gb300 import inputs, obem

pytestmark = pytest.mark.gpu
QE, ME = 1.602176634e-19, 9.1093837015e-31
INTS = ["n_after", "spawned_pairs", "absorbed", "attached", "recombined_pairs", "collisions", "trials", "n_electron",
        "n_cation", "n_anion"]


def _charges(rng, n):
    ch = inputs.avalanche_snapshot(rng, n, gap=1e-3)
    ch.pos_q[:, 2] = np.clip(ch.pos_q[:, 2], 5e-5, 9.5e-4)
    e = ch.species == 0
    d = rng.normal(size=(int(e.sum()), 3))
    d *= (np.sqrt(2 * 50 * QE / ME) / np.linalg.norm(d, axis=1))[:, None]
    ch.vel[e, :3] = d.astype(np.float32)                    # 50 eV: ionisations in every step
    return ch


def _track(cap, ch, steps=3):
    ctx = obem.obem_create(capacity=cap, dt=1e-12, seed=7, z_lo=0.0, z_hi=1e-3, beta=1e-13, softening=1e-9, flags=0,
                           e_ext=(0.0, 0.0, -1e6))
    try:
        obem.obem_gas_load(ctx, inputs.argon_like_gas())
        st, stats, out = obem.DeviceState(cap), obem.new_stats(), []
        st.upload(ch)
        for s in range(steps):
            obem.obem_step(ctx, st, s, stats)
            torch.cuda.synchronize()
            out.append(obem.read_stats(stats))
        return st.download(), out
    finally:
        obem.obem_destroy(ctx)


@pytest.mark.parametrize("cap", [16385, 65536, 65537, 524288, 524289])
def test_step_is_the_same_for_every_capacity(cap):
    ch = _charges(np.random.default_rng(11), 5001)
    (a, ida), sa = _track(16384, ch)
    (b, idb), sb = _track(cap, ch)
    assert ida == idb and a.n == b.n and a.n > 5001
    for k in ("pos_q", "vel", "id", "birth", "species"):
        assert np.array_equal(getattr(a, k), getattr(b, k)), k
    for x, y in zip(sa, sb):
        assert [x[k] for k in INTS] == [y[k] for k in INTS]
    # the moments are FP64 sums of ~1e4 terms in another order: n 2^-53 of sum |x|
    el = b.pos_q[b.species == 0, :3].astype(np.float64)
    for s in (sa[-1], sb[-1]):
        assert np.all(np.abs(np.asarray(s["sum_e"]) - el.sum(0)) <= 1e-12 * np.abs(el).sum(0))


@pytest.mark.parametrize("caps", [(101_000, 3000), (200_000, 3000), (380_000, 3000)])
def test_batch_units(caps):
    """4,900, 19,600 and 69,000 tile pairs: units of 1, 4 and 16."""
    rng = np.random.default_rng(caps[0])
    chs = [_charges(rng, n) for n in (2500, 1025)]
    ctx = obem.obem_create(capacity=16, dt=1e-12, softening=1e-9, flags=obem.OBEM_STEP_SPACE_CHARGE)
    try:
        obem.obem_gas_load(ctx, inputs.argon_like_gas())
        b = obem.Batch(ctx, list(caps), [0.0, 0.0], [1e-3, 1e-3], [1, 2])
        try:
            st = b.state()
            st.upload(chs)
            out = torch.full((st.capacity, 4), float("nan"), device="cuda")
            b.field_eval(st, out)
            torch.cuda.synchronize()
            for c, ch in enumerate(chs):
                o = int(b.seg_off[c])
                got = out[o:o + len(ch.pos_q)].cpu().numpy()
                E, _ = oracle.nbody_field(ch.pos_q[:, :3].astype(np.float64), ch.pos_q.astype(np.float64), True, 1e-9)
                assert guarded_rel_err(got[:, :3], E) <= FIELD_TOL
        finally:
            b.destroy()
    finally:
        obem.obem_destroy(ctx)
