"""The FP32 GEMM with unit-stride operands against FP64 products and against the general-stride kernel."""
import pytest
import torch

pytestmark = pytest.mark.gpu

# edges of the 16 x 32, 32 x 32 and 32 x 64 tiles and of the 32-step stages; rows of every copy width
SHAPES = [(1, 1, 1), (3, 5, 2), (16, 32, 32), (17, 33, 31), (32, 256, 418), (31, 255, 33), (512, 101, 512),
          (513, 101, 274), (512, 512, 64), (545, 511, 37), (1024, 12, 96), (64, 8, 2593)]


def _operand(rows, k, kmajor, g, pad):
    """A [rows, k] view with a unit stride along k (kmajor) or along the rows, `pad` elements past a row."""
    buf = torch.randn(rows if kmajor else k, (k if kmajor else rows) + pad, generator=g).cuda()
    return buf[:, :k] if kmajor else buf[:, :rows].t()


def _general(t):
    """The same values with no unit stride."""
    buf = torch.empty(t.shape[0], t.shape[1], 2, device=t.device)
    buf[:, :, 0] = t
    return buf[:, :, 0]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
def test_gemm_f32_unit_strides(M, N, K, a_k, b_k):
    from paper_2602_21203_gb300 import ops
    g = torch.Generator().manual_seed(M * 31 + N * 7 + K + 2 * a_k + b_k)
    pad = (M + N + K) % 3
    A, B = _operand(M, K, a_k, g, pad), _operand(N, K, b_k, g, 0)
    bias = torch.randn(N, generator=g).cuda()
    C0 = torch.randn(M, N, generator=g).cuda()
    out = ops.gemm(A, B, bias=bias)
    acc = ops.gemm(A, B, out=C0.clone(), accumulate=True)
    # one rounding per fused multiply-add and one for the bias: |error| <= (K + 1) u (|A| |B|^T + |bias|), u = 2^-24
    exact = A.double() @ B.double().t() + bias.double()
    bound = (K + 1) * 2.0 ** -24 * (A.double().abs() @ B.double().abs().t() + bias.double().abs()) * 1.01
    assert bool(((out.double() - exact).abs() <= bound).all())
    # the general kernel accumulates in the same order: the same bits
    if K > 1 and M > 1 and N > 1:
        assert torch.equal(out, ops.gemm(_general(A), _general(B), bias=bias))
        assert torch.equal(acc, ops.gemm(_general(A), _general(B), out=C0.clone(), accumulate=True))


def test_gemm_f32_non_finite_values_stay_in_their_rows():
    from paper_2602_21203_gb300 import ops
    A, B = torch.randn(33, 40).cuda(), torch.randn(65, 40).cuda()
    A[32, 39], B[64, 0] = float("inf"), float("nan")
    out = ops.gemm(A, B)
    assert bool(torch.isfinite(out[:32, :64]).all())
    assert torch.equal(torch.nan_to_num(out, 7.0), torch.nan_to_num(ops.gemm(_general(A), _general(B)), 7.0))


# both sides of the lines between this kernel and the general one: grids of 465, 496, 722, 1,170 and 2,574 tiles, the last
# K that changes sides and the next, rows copied 16, 8 and 4 bytes at a time
@pytest.mark.parametrize("M,N,K", [(992, 960, 33), (992, 1024, 48), (992, 1024, 49), (992, 1024, 101), (1200, 1200, 33), (1200, 1200, 34),
                                   (2080, 1100, 16), (2080, 1100, 48), (2080, 1100, 49), (2080, 1100, 71), (2081, 2494, 130),
                                   (2081, 2494, 141), (2081, 2494, 201)])
@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
def test_gemm_f32_large_grids(M, N, K, a_k, b_k):
    test_gemm_f32_unit_strides(M, N, K, a_k, b_k)
