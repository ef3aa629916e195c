"""The tensor-core update C -= A B at the sizes where its kernel and tile
change: K up to 128 from the FP32 operands (tiles of 64 or 128 columns, 16-byte
loads when both operands are aligned), then 128 x 128 and 256 x 256 tiles fed by
TMA; remainders of rows, columns and K, blocks inside larger arrays."""
import pytest
import torch

from paper_2110_09214_gb300 import obem

pytestmark = pytest.mark.gpu


def _bf16(t):
    return t.to(torch.bfloat16).to(torch.float64)


# (FP32 accumulation of exact BF16 products: a sum of K <= 1200 terms in any
# order is within 1200 x 2^-24 = 7e-5 of sum |a b| at worst, within a few
# sqrt(1200) x 2^-24 = 2e-6 for these random signs; 3e-5 separates both from a
# misplaced 1 in 1200 terms, about 1e-3.)
@pytest.mark.parametrize("off", [4, 3])
@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (127, 63, 63), (129, 65, 64), (128, 64, 65), (3001, 64, 128),
                                   (257, 20001, 127), (1700, 1700, 128), (300, 300, 129), (2049, 300, 257),
                                   (1500, 1700, 1025), (260, 2300, 1030)])
def test_update(M, N, K, off):
    g = torch.Generator().manual_seed(M + 3 * N + 7 * K + off)
    C0 = torch.randn(M + 2, (N + off + 7) // 4 * 4, generator=g)
    A = torch.randn(M, (K + off + 7) // 4 * 4, generator=g).cuda()[:, off:off + K]
    B = torch.randn(K, (N + off + 7) // 4 * 4, generator=g).cuda()[:, off:off + N]
    C = C0.cuda()
    ctx = obem.obem_create(capacity=8, dt=1e-12)
    try:
        obem.obem_tc_gemm(ctx, C[1:1 + M, off:off + N], A, B)
        torch.cuda.synchronize()
    finally:
        obem.obem_destroy(ctx)
    a, b, c = _bf16(A), _bf16(B), C0.cuda().double()[1:1 + M, off:off + N]
    err = ((C[1:1 + M, off:off + N].double() - (c - a @ b)).abs() / (c.abs() + a.abs() @ b.abs())).max().item()
    assert err <= 3e-5, err
    C[1:1 + M, off:off + N] = C0.cuda()[1:1 + M, off:off + N]
    assert torch.equal(C, C0.cuda())
