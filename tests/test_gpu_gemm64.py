"""The unsplit BF16 GEMM (128 x 64 tiles) at the edges of its tiles, against FP64 products of the same operands."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def _operand(rows, k, kmajor, g):
    """A [rows, k] BF16 view, K-major or MN-major, with the 8-element row padding the tensor maps need."""
    r, c = (rows, k) if kmajor else (k, rows)
    buf = torch.randn(r, (c + 7) // 8 * 8, generator=g).to(torch.bfloat16).cuda()
    return buf[:, :c] if kmajor else buf[:, :c].t()


@pytest.mark.parametrize("M,N,K", [(1, 1, 1), (128, 64, 64), (127, 63, 65), (129, 65, 256), (257, 101, 130), (33, 127, 512),
                                   (8, 129, 320), (512, 512, 512), (640, 200, 383), (4096, 12, 64)])
@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
def test_gemm64(M, N, K, a_k, b_k):
    from paper_2602_21203_gb300 import ops
    g = torch.Generator().manual_seed(M + 3 * N + 7 * K + 2 * a_k + b_k)
    A, B = _operand(M, K, a_k, g), _operand(N, K, b_k, g)
    bias = torch.randn(N, generator=g).cuda()
    exact = A.double() @ B.double().t()
    # BF16 products are exact in FP32; K additions of at most 2^-22 relative error each (truncating adders included)
    bound = (K + 2) * 2.0 ** -22 * (A.double().abs() @ B.double().abs().t() + bias.double().abs()) + 1e-30
    out = ops.gemm(A, B, bias=bias)
    assert bool(((out.double() - exact - bias.double()).abs() <= bound).all())
    # the products alone, then accumulated onto rows wider than the tile: neighbours stay as they were
    plain = ops.gemm(A, B)
    wide = torch.full((M, N + 3), 2.0, device="cuda")
    ops.gemm(A, B, out=wide[:, 1:N + 1], accumulate=True)
    assert torch.equal(wide[:, 1:N + 1], 2.0 + plain)
    assert bool((wide[:, 0] == 2).all()) and bool((wide[:, N + 1:] == 2).all())
