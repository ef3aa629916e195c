"""The tracking step of few charges in a large state: the chunks follow the live
count, and the state is bit for bit that of a context of the set's own size."""
import numpy as np
import pytest
import torch

from paper_2110_09214_gb300 import inputs, obem

pytestmark = pytest.mark.gpu
E = 1.602176634e-19


def _charges(n):
    rng = np.random.default_rng(n)
    ch = inputs.avalanche_snapshot(rng, n, gap=2e-3)
    ch.pos_q[:, 2] = np.clip(ch.pos_q[:, 2], 4e-5, 1.96e-3)
    hot = rng.random(n) < 0.2                               # 50 eV electrons: ionisations in the first step
    e = (ch.species == inputs.SP_ELECTRON) & hot
    d = rng.normal(size=(int(e.sum()), 3))
    d /= np.linalg.norm(d, axis=1)[:, None]
    ch.vel[e, :3] = d * np.sqrt(2 * 50 * E / inputs.M_ELECTRON)
    return ch


def _run(ch, cap, steps):
    ctx = obem.obem_create(capacity=cap, dt=1e-12, seed=7, softening=1e-9, z_lo=0.0, z_hi=2e-3, beta=1e-13, flags=0)
    try:
        obem.obem_gas_load(ctx, inputs.argon_like_gas())
        st = obem.DeviceState(cap)
        st.upload(ch)
        Ein = torch.zeros((cap, 4), device="cuda")
        Ein[:, 2] = 1e6
        stats = obem.new_stats()
        out = []
        for k in range(steps):
            obem.obem_step(ctx, st, k, stats, E_in=Ein)
            s = obem.read_stats(stats)
            assert s["status"] == 0
            out.append({q: s[q] for q in ("n_after", "spawned_pairs", "absorbed", "attached", "recombined_pairs",
                                          "collisions", "trials", "n_electron", "n_cation", "n_anion")})
        return st.download(), out
    finally:
        obem.obem_destroy(ctx)


@pytest.mark.parametrize("n", [1, 5, 1000, 16_384, 16_385, 65_536, 65_537])
def test_state_does_not_depend_on_the_capacity(n):
    ch = _charges(n)
    (a, na), sa = _run(ch, 2 * n + 64, 3)
    (b, nb), sb = _run(ch, 600_000, 3)
    assert sa == sb and na == nb and a.n == b.n
    if n >= 1000:
        assert sa[0]["spawned_pairs"] > 0
    for f in ("pos_q", "vel"):
        assert np.array_equal(getattr(a, f).view(np.uint32), getattr(b, f).view(np.uint32)), f
    for f in ("id", "birth", "species"):
        assert np.array_equal(getattr(a, f), getattr(b, f)), f
