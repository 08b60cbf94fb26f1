"""The FP32 GEMM with unit-stride operands against FP64 products and against the general-stride kernel."""
import ctypes

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


def _tile(*shapes):
    """The output tile launch_layout (sq_gemm_f32.cu) gives a launch of these (M, N)."""
    tiles = lambda bm, bn: sum(-(-m // bm) * -(-n // bn) for m, n, *_ in shapes)
    return (32, 64) if tiles(32, 64) >= 100 else (32, 32) if tiles(32, 32) >= 100 else (16, 32)


@pytest.mark.parametrize("M,N,K", [(512, 256, 130), (513, 255, 37), (1000, 97, 64), (31, 3200, 5)])
@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
def test_gemm_f32_middle_tile(M, N, K, a_k, b_k):
    assert _tile((M, N)) == (32, 32)
    test_gemm_f32_unit_strides(M, N, K, a_k, b_k)


class _Problem(ctypes.Structure):
    """sq::GemmProblem (sq_kernels.cuh)."""
    _fields_ = [("M", ctypes.c_int), ("N", ctypes.c_int), ("K", ctypes.c_int),
                ("A", ctypes.c_void_p), ("sa_m", ctypes.c_int64), ("sa_k", ctypes.c_int64),
                ("B", ctypes.c_void_p), ("sb_n", ctypes.c_int64), ("sb_k", ctypes.c_int64),
                ("C", ctypes.c_void_p), ("sc_m", ctypes.c_int64), ("sc_n", ctypes.c_int64),
                ("bias", ctypes.c_void_p), ("mask", ctypes.c_void_p), ("sm_m", ctypes.c_int64), ("sm_n", ctypes.c_int64),
                ("accumulate", ctypes.c_int), ("n_sum", ctypes.c_int), ("a_sum", ctypes.c_int64), ("b_sum", ctypes.c_int64)]


# several problems of one launch (more than one batch of them too), each the sum of n_sum operand pairs a distance
# apart that leaves copies of 16, 8 and 4 bytes, with steps of K that end inside a stage, masks and accumulation
@pytest.mark.parametrize("shapes,n_sum,gap,tile", [([(33, 65, 37), (512, 20, 64)], 2, 0, (16, 32)),
                                                   ([(33, 65, 37), (130, 12, 96), (5, 256, 1)], 2, 2, (16, 32)),
                                                   ([(512, 101, 70), (513, 101, 33), (1, 1, 1)], 3, 1, (32, 32)),
                                                   ([(512, 300, 40), (700, 129, 34)], 2, 4, (32, 64)),
                                                   ([(40 + i, 30 + i, 20 + i) for i in range(11)], 1, 0, (16, 32))])
@pytest.mark.parametrize("a_k,b_k", [(True, True), (True, False), (False, True), (False, False)])
def test_gemm_f32_grouped_sums(shapes, n_sum, gap, tile, a_k, b_k):
    from paper_2602_21203_gb300 import lib, ops
    assert _tile(*shapes[:8]) == tile
    g = torch.Generator().manual_seed(len(shapes) + 10 * gap + 2 * a_k + b_k)
    probs, want, outs, keep = (_Problem * len(shapes))(), [], [], []
    for i, (M, N, K) in enumerate(shapes):
        ld = {True: (K + 3) // 4 * 4, False: (M + 3) // 4 * 4}[a_k], {True: (K + 3) // 4 * 4, False: (N + 3) // 4 * 4}[b_k]
        dist = ld[0] * (M if a_k else K) + gap, ld[1] * (N if b_k else K) + gap
        bufs = [torch.randn(n_sum * d, generator=g).cuda() for d in dist]

        def pair(j, q, rows, kmajor):
            st = (ld[j], 1) if kmajor else (1, ld[j])
            return bufs[j].as_strided((rows, K), st, q * dist[j])
        A, B = [pair(0, q, M, a_k) for q in range(n_sum)], [pair(1, q, N, b_k) for q in range(n_sum)]
        bias, mask = torch.randn(N, generator=g).cuda(), torch.randn(M, N, generator=g).cuda()
        C = torch.randn(M, N, generator=g).cuda()
        v = torch.where(mask > 0, ops.gemm(torch.cat(A, 1), torch.cat(B, 1), bias=bias), torch.zeros_like(C))
        want.append(C + v if i % 2 else v)      # one chain over the pairs in turn: the bits of the pairs side by side
        P = probs[i]
        P.M, P.N, P.K, P.A, P.B, P.C = M, N, K, bufs[0].data_ptr(), bufs[1].data_ptr(), C.data_ptr()
        P.sa_m, P.sa_k = (ld[0], 1) if a_k else (1, ld[0])
        P.sb_n, P.sb_k = (ld[1], 1) if b_k else (1, ld[1])
        P.sc_m, P.sc_n, P.bias, P.mask, P.sm_m, P.sm_n = N, 1, bias.data_ptr(), mask.data_ptr(), N, 1
        P.accumulate, P.n_sum, P.a_sum, P.b_sum = i % 2, n_sum, dist[0], dist[1]
        outs.append(C)
        keep.append((bufs, bias, mask))
    f = lib.load()["_ZN2sq15launch_gemm_f32EPKNS_11GemmProblemEiP11CUstream_st"]
    f.argtypes, f.restype = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p], ctypes.c_bool
    assert f(probs, len(shapes), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    for C, w in zip(outs, want):
        assert torch.equal(C, w)
