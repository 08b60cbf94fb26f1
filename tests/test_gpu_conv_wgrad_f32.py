"""The FP32 convolutions' weight gradient over row groups of four pixels, against the FP64 kernel."""
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
# n, cin, cout, h, w, stride: rows of 1 to 5 and of 7, 20 and 39 pixels (every remainder of a group), splits
# that start and end inside rows, many images a stage, channel counts around 4, 8, 16 and 32, both strides
SHAPES = [(300, 16, 16, 4, 6, 1), (200, 1, 1, 3, 4, 1), (61, 17, 32, 20, 9, 1), (33, 33, 33, 9, 7, 1), (9, 20, 33, 12, 41, 2),
          (70, 4, 8, 6, 8, 2), (129, 3, 16, 5, 11, 2), (2, 32, 32, 40, 22, 1), (90, 5, 40, 8, 5, 1), (400, 2, 3, 3, 3, 1)]


@pytest.mark.parametrize("n,cin,cout,h,w,s", SHAPES)
def test_conv_wgrad_f32_matches_fp64(n, cin, cout, h, w, s):
    from paper_2602_21203_gb300 import ops
    g = torch.Generator().manual_seed(n + 3 * cin + 5 * cout + 7 * h + 11 * w + s)
    oh, ow = (h - 3) // s + 1, (w - 3) // s + 1
    x, wt = torch.randn(n, cin, h, w, generator=g).cuda(), torch.randn(cout, cin, 3, 3, generator=g).cuda()
    dy = torch.randn(n, cout, oh, ow, generator=g).cuda()
    _, dw, db = ops.conv3x3_bwd(x, wt, dy, s)
    _, dwd, dbd = ops.conv3x3_bwd(x.double(), wt.double(), dy.double(), s)
    _, bw, bb = ops.conv3x3_bwd(x.double().abs(), wt.double().abs(), dy.double().abs(), s)
    # chains of at most k fused multiply-adds and the sum of their results: at most k + 64 roundings
    bound = (n * oh * ow + 64) * U * 1.01
    assert bool(((dw.double() - dwd).abs() <= bound * bw).all())
    assert bool(((db.double() - dbd).abs() <= bound * bb).all())
    # an infinite corner reaches the one tap that reads it, and no other product of its group
    x[0, 0, 0, 0] = float("inf")
    dy[0, :, 0, 0] = 1.0
    _, dwi, dbi = ops.conv3x3_bwd(x, wt, dy, s)
    assert bool(torch.isinf(dwi[:, 0, 0, 0]).all()) and bool(torch.isfinite(dbi).all())
    dwi[:, 0, 0, 0] = 0
    assert bool(torch.isfinite(dwi).all())
