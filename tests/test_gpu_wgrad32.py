"""The tensor-core weight gradient of a 32 -> 32 channel layer over its staging edges, against FP64."""
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _case(n, H, W):
    from paper_2602_21203_gb300 import ops
    g = torch.Generator().manual_seed(n + 3 * H + 5 * W)
    x = torch.randn(n, 32, H, W, generator=g).bfloat16().float().cuda()
    dy = torch.randn(n, 32, H - 2, W - 2, generator=g).bfloat16().float().cuda()
    return x, dy, ops.to_phwc(x), ops.to_phwc(dy)


def _check(dw, db, x, dy):
    from paper_2602_21203_gb300 import ops
    zero = torch.zeros(32, 32, 3, 3, device="cuda", dtype=torch.float64)
    _, rw, rb = ops.conv3x3_bwd(x.double(), zero, dy.double(), 1)
    _, bw, bb = ops.conv3x3_bwd(x.double().abs(), zero, dy.double().abs(), 1)
    # products of BF16 values are exact in FP32; every addition errs by at most 2 u of the running sum
    tol = (dy.shape[0] * dy.shape[2] * dy.shape[3] + 160) * 2 * U * 1.01
    assert bool(((dw.double() - rw).abs() <= tol * bw).all())
    assert bool(((db.double() - rb).abs() <= tol * bb).all())


# one image and one pixel; one to five images a CTA, the last CTA short; K that fills its last 16 pixels
# or not; an image too large for the padded pitch
@pytest.mark.parametrize("n,H,W", [(1, 3, 3), (5, 4, 3), (149, 7, 6), (297, 9, 16), (740, 5, 5), (3, 18, 12), (2, 23, 15), (2, 17, 18)])
def test_wgrad32(n, H, W):
    from paper_2602_21203_gb300 import ops
    x, dy, xp, dyp = _case(n, H, W)
    _check(*ops.wgrad32(xp, dyp, H, W), x, dy)


def test_wgrad32_workspace_of_any_alignment():
    from paper_2602_21203_gb300 import lib, ops
    x, dy, xp, dyp = _case(9, 8, 7)
    L = lib.load()
    nb = L.squint_op_wgrad32_workspace(9)
    buf = torch.empty(nb + 4, dtype=torch.uint8, device="cuda")
    dw, db = torch.empty(32, 32, 3, 3, device="cuda"), torch.empty(32, device="cuda")
    s = torch.cuda.current_stream().cuda_stream
    assert L.squint_op_wgrad32(9, 8, 7, xp.data_ptr(), dyp.data_ptr(), dw.data_ptr(), db.data_ptr(), buf.data_ptr() + 4, nb, s) == 0
    torch.cuda.synchronize()
    _check(dw, db, x, dy)
    rw, rb = ops.wgrad32(xp, dyp, 8, 7)
    assert torch.equal(dw, rw) and torch.equal(db, rb)


def test_wgrad32_images_do_not_mix():
    """A NaN in the image behind the last one used, where the last rows of a slot lie, stays out."""
    from paper_2602_21203_gb300 import ops
    x, dy, xp, dyp = _case(4, 6, 9)
    want = ops.wgrad32(xp[:3].contiguous(), dyp[:3].contiguous(), 6, 9)
    big = torch.full_like(xp, float("nan"))
    big[:3] = xp[:3]
    got = ops.wgrad32(big[:3], dyp[:3], 6, 9)
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
