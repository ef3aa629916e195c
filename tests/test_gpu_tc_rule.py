"""The tensor-core update C -= A B of short K on both sides of the size of C up
to which it runs from the FP32 operands in one kernel."""
import pytest
import torch

from paper_2110_09214_gb300 import obem

pytestmark = pytest.mark.gpu


# FP32 accumulation of at most 128 exact products of BF16 numbers is within 128 x
# 2^-24 = 7.7e-6 of sum |a b|, the subtraction from C within 2^-24 of |C|: 1e-5.
@pytest.mark.parametrize("off", [4, 3])
@pytest.mark.parametrize("M,N,K", [(10_000, 1000, 64), (10_000, 1001, 64), (3201, 3301, 1), (129, 80_000, 65), (80_001, 129, 127),
                                   (3200, 3200, 128), (4000, 2600, 8), (20_001, 515, 33)])
def test_short_k(M, N, K, off):
    g = torch.Generator(device="cuda").manual_seed(M + 3 * N + 7 * K + off)
    rnd = lambda r, c: torch.randn(r, (c + off + 7) // 4 * 4, generator=g, device="cuda")  # noqa: E731
    C0, A, B = rnd(M + 2, N), rnd(M, K)[:, off:off + K], rnd(K, N)[:, off:off + N]
    C = C0.clone()
    ctx = obem.obem_create(capacity=8, dt=1e-12)
    try:
        obem.obem_tc_gemm(ctx, C[1:1 + M, off:off + N], A, B)
        torch.cuda.synchronize()
    finally:
        obem.obem_destroy(ctx)
    a, b, c = A.to(torch.bfloat16).double(), B.to(torch.bfloat16).double(), C0[1:1 + M, off:off + N].double()
    err = ((C[1:1 + M, off:off + N].double() - (c - a @ b)).abs() / (c.abs() + a.abs() @ b.abs())).max().item()
    assert err <= 1e-5, err
    C[1:1 + M, off:off + N] = C0[1:1 + M, off:off + N]
    assert torch.equal(C, C0)
