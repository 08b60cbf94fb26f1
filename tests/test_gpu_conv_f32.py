"""The FP32 convolutions (forward, data and weight gradient) against the FP64 kernels on the same values."""
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -24
# n, cin, cout, h, w, stride: tiles that end inside rows, at row ends and across images; one-pixel
# images; channel counts around 4, 8 and 32; every pixel count a thread; a region too wide for the
# staged kernels (the last one, which the general kernels take)
SHAPES = [(1, 1, 1, 3, 3, 1), (5, 3, 16, 16, 16, 2), (32, 16, 16, 7, 7, 1), (70, 2, 3, 3, 3, 1), (3, 4, 8, 9, 12, 1),
          (2, 5, 33, 21, 10, 2), (7, 9, 31, 9, 33, 3), (150, 32, 32, 15, 15, 1), (40, 33, 40, 13, 8, 1),
          (90, 8, 24, 11, 11, 1), (2, 3, 32, 32, 32, 2), (3, 6, 7, 10, 10, 5), (1, 2, 4, 5, 700, 1)]


def _inputs(n, cin, cout, h, w, s):
    g = torch.Generator().manual_seed(n + 3 * cin + 5 * cout + 7 * h + 11 * w + s)
    oh, ow = (h - 3) // s + 1, (w - 3) // s + 1
    x, wt = torch.randn(n, cin, h, w, generator=g).cuda(), torch.randn(cout, cin, 3, 3, generator=g).cuda()
    return x, wt, torch.randn(cout, generator=g).cuda(), torch.randn(n, cout, oh, ow, generator=g).cuda()


@pytest.mark.parametrize("n,cin,cout,h,w,s", SHAPES)
def test_conv_f32_matches_fp64(n, cin, cout, h, w, s):
    from paper_2602_21203_gb300 import ops
    x, wt, b, dy = _inputs(n, cin, cout, h, w, s)
    xd, wd, bd, dyd = (t.double() for t in (x, wt, b, dy))
    # a chain of k fused multiply-adds errs by at most k u (sum of |products|); 1.01 for the bound's own second order
    y = ops.conv3x3_fwd(x, wt, b, s, False)
    bound = (cin * 9 + 1) * U * 1.01 * ops.conv3x3_fwd(xd.abs(), wd.abs(), bd.abs(), s, False)
    assert bool(((y.double() - ops.conv3x3_fwd(xd, wd, bd, s, False)).abs() <= bound).all())
    yr = ops.conv3x3_fwd(x, wt, b, s, True)
    assert torch.equal(yr, torch.relu(y))
    mask = torch.randn(x.shape, generator=torch.Generator().manual_seed(1)).cuda()
    dx, dw, db = ops.conv3x3_bwd(x, wt, dy, s)
    dxm, dwm, dbm = ops.conv3x3_bwd(x, wt, dy, s, dx_mask=mask)
    assert torch.equal(dxm, torch.where(mask > 0, dx, torch.zeros_like(dx))) and torch.equal(dw, dwm) and torch.equal(db, dbm)
    dxd, dwd, dbd = ops.conv3x3_bwd(xd, wd, dyd, s)
    bx, bw, bb = ops.conv3x3_bwd(xd.abs(), wd.abs(), dyd.abs(), s)
    assert bool(((dx.double() - dxd).abs() <= cout * 9 * U * 1.01 * bx).all())
    pixels = dy.shape[0] * dy.shape[2] * dy.shape[3]
    assert bool(((dw.double() - dwd).abs() <= pixels * U * 1.01 * bw).all())
    assert bool(((db.double() - dbd).abs() <= pixels * U * 1.01 * bb).all())


def test_conv_f32_images_do_not_mix():
    """NaN and infinity in one image reach that image's outputs alone."""
    from paper_2602_21203_gb300 import ops
    x, wt, b, _ = _inputs(6, 5, 9, 9, 11, 1)
    clean = ops.conv3x3_fwd(x, wt, b, 1, True)
    x[3, :, 4, 4] = float("nan")
    x[5, 2, 8, 10] = float("inf")
    y = ops.conv3x3_fwd(x, wt, b, 1, False)
    keep = [0, 1, 2, 4]
    assert torch.equal(torch.relu(y[keep]), clean[keep])
    assert bool(torch.isnan(y[3, :, 2:5, 2:5]).all()) and not bool(torch.isnan(y[3, :, :2]).any())


# grids on both sides of the line from which one input channel, or few and a wide stride, take the general kernel
@pytest.mark.parametrize("n,cin,cout,h,w,s", [(1032, 1, 8, 21, 22, 2), (1020, 1, 8, 21, 22, 2), (1030, 2, 8, 21, 22, 2),
                                              (530, 8, 40, 30, 32, 3), (500, 8, 40, 30, 32, 3), (530, 9, 40, 30, 32, 3)])
def test_conv_f32_few_channels(n, cin, cout, h, w, s):
    test_conv_f32_matches_fp64(n, cin, cout, h, w, s)


SMEM = 48 * 1024


def _plan(n, channels, oh, ow, rs, pw):
    """Pixels a thread and stages of launch_conv (sq_conv_f32.cu) for n images of oh x ow outputs read from rows pw wide."""
    m, p = n * oh * ow, 4
    while p > 1 and -(-m // (32 * p)) * -(-channels // 32) < 2 * 152:
        p //= 2
    px = 32 * p
    words = ((-(-(px - 1) // ow) + 1) * rs + max(0, 3 - rs) * (-(-(px - 1) // (oh * ow)) + 1)) * pw
    stage, table = 4 * (4 * 9 * 36 + 4 * words), 4 * words
    assert 2 * stage + table <= SMEM
    return p, 3 if 3 * stage + table <= SMEM else 2


# four pixels a thread, forward and data gradient, where the multiplying warps stage too: the training layer; output
# channels that are no multiple of 8 and one warp of input channels; stride 2 with an input row that no tap reads;
# rows so wide that two stages fit; last tiles of one to four pixels a lane
@pytest.mark.parametrize("n,cin,cout,h,w,s,stages", [(300, 32, 32, 15, 15, 1, (3, 3)), (200, 5, 44, 17, 13, 1, (3, 3)),
                                                     (700, 3, 20, 18, 21, 2, (2, 3)), (12, 6, 9, 30, 120, 1, (2, 2)),
                                                     (4325, 7, 32, 5, 5, 1, (3, 3))])
def test_conv_f32_four_pixels_a_thread(n, cin, cout, h, w, s, stages):
    oh, ow = (h - 3) // s + 1, (w - 3) // s + 1
    assert _plan(n, cout, oh, ow, s, w) == (4, stages[0]) and _plan(n, cin, h, w, 1, w + 2) == (4, stages[1])
    test_conv_f32_matches_fp64(n, cin, cout, h, w, s)


@pytest.mark.parametrize("n,cin,cout,h,w,s,p", [(150, 12, 32, 15, 15, 1, 2), (100, 32, 7, 21, 19, 2, 1), (3, 40, 33, 11, 12, 1, 1)])
def test_conv_f32_fewer_pixels_a_thread(n, cin, cout, h, w, s, p):
    oh, ow = (h - 3) // s + 1, (w - 3) // s + 1
    assert _plan(n, cout, oh, ow, s, w)[0] == p
    test_conv_f32_matches_fp64(n, cin, cout, h, w, s)
