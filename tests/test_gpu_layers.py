"""The one-call layer operations against the single operations they are made of."""
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


def _rand(*shape, seed):
    return torch.randn(*shape, generator=torch.Generator().manual_seed(seed)).cuda()


def _dirty():
    """Leave NaN in the memory that the next allocations take."""
    junk = torch.full((1 << 22,), float("nan"), device="cuda")
    del junk


def _sum_close(got, t, rows):
    """Column sums in any order: (rows - 1) additions, each rounded once."""
    exact, bound = t.double().sum(0), rows * U * t.double().abs().sum(0) * 1.01
    assert bool(((got.double() - exact).abs() <= bound).all())


# rows of 16-byte chunks and not, one element, pad columns, views with a row stride, offsets of 4 and 8 bytes
@pytest.mark.parametrize("rows,cols,ld,off", [(1, 1, 1, 0), (7, 8, 8, 0), (9, 13, 13, 0), (16, 130, 132, 0), (33, 274, 274, 0),
                                              (5, 516, 520, 4), (5, 516, 520, 1), (8, 2592, 2592, 0), (3, 31, 40, 2)])
def test_cast_rows(rows, cols, ld, off):
    from paper_2602_21203_gb300 import ops
    buf = _rand(rows * ld + off, seed=rows + cols)
    x = buf[off:].view(rows, ld)[:, :cols]
    _dirty()
    y = ops.cast_bf16(x)
    assert torch.equal(y, x.to(torch.bfloat16))
    pad = y.as_strided((rows, y.stride(0)), (y.stride(0), 1))[:, cols:]
    assert bool((pad == 0).all())


@pytest.mark.parametrize("M,K,N", [(1, 1, 1), (31, 13, 7), (32, 18, 12), (33, 274, 101), (64, 96, 128), (129, 130, 132), (900, 70, 33)])
@pytest.mark.parametrize("strided", [False, True])
def test_linear_layers(M, K, N, strided):
    from paper_2602_21203_gb300 import ops
    x, w, b, dy = (_rand(M, 2 * K, seed=1)[:, :K] if strided else _rand(M, K, seed=1), _rand(N, K, seed=2), _rand(N, seed=3),
                   _rand(M, N, seed=4))
    xh, wh, dyh = ops.cast_bf16(x), ops.cast_bf16(w), ops.cast_bf16(dy)
    _dirty()
    y, xs, ws = ops.linear_bf16_fwd(x, w, b)
    assert torch.equal(y, ops.gemm(xh, wh, bias=b)) and torch.equal(xs, xh) and torch.equal(ws, wh)
    dx, dw, db = ops.linear_bf16_bwd(dy, xs, ws)
    assert torch.equal(dx, ops.gemm(dyh, wh.t(), M=M, N=K, K=N))
    assert torch.equal(dw, ops.gemm(dyh.t(), xh.t(), M=N, N=K, K=M))
    _sum_close(db, dy, M)
    assert ops.linear_bf16_bwd(dy, xs, ws, (False, False, True))[:2] == (None, None)
    dx, dw, db = ops.linear_bwd(dy, x, w)
    assert torch.equal(dx, ops.gemm(dy, w.t(), M=M, N=K, K=N)) and torch.equal(dw, ops.gemm(dy.t(), x.t(), M=N, N=K, K=M))
    _sum_close(db, dy, M)


@pytest.mark.parametrize("M,kin,H,nh,nout", [(1, 5, 32, 1, 1), (33, 18, 64, 2, 12), (130, 274, 256, 3, 101), (800, 40, 128, 2, 51)])
def test_mlp_head_layer(M, kin, H, nh, nout):
    from paper_2602_21203_gb300 import ops
    dims = [kin] + [H] * nh + [nout]
    ws = [_rand(b, a, seed=i) / a ** 0.5 for i, (a, b) in enumerate(zip(dims, dims[1:]))]
    bs = [_rand(n, seed=10 + i) * 0.1 for i, n in enumerate(dims[1:])]
    gs, betas = [1 + 0.1 * _rand(H, seed=20 + i) for i in range(nh)], [0.1 * _rand(H, seed=30 + i) for i in range(nh)]
    x, dout = _rand(M, kin, seed=40), _rand(M, nout, seed=41) / M
    wh = [ops.cast_bf16(w) for w in ws]
    ref, sv = ops.mlp_bf16(ops.cast_bf16(x), wh, bs, gs, betas)
    _dirty()
    out, saved = ops.mlp_head_fwd(x, ws, bs, gs, betas)
    assert torch.equal(out, ref)
    for l in range(nh):
        for got, want in zip((saved[2][l], saved[3][l], saved[4][l], saved[5][0, l], saved[5][1, l]), sv[l]):
            assert torch.equal(got, want)
    _dirty()
    dx, dws, dbs, dgs, dbetas = ops.mlp_head_bwd(dout, gs, saved, kin)
    dy = dout
    for l in range(nh, -1, -1):
        h = ops.cast_bf16(x) if l == 0 else sv[l - 1][2]
        dyh = ops.cast_bf16(dy)
        want = ops.gemm(dyh.t(), h.t(), M=dims[l + 1], N=dims[l], K=M)
        # the layers' weight gradients are one launch, whose K split may differ: M additions in another order
        bound = 2 * M * 2.0 ** -22 * (dyh.double().abs().t() @ h.double().abs()) + 1e-30
        assert bool(((dws[l].double() - want.double()).abs() <= bound).all())
        _sum_close(dbs[l], dy, M)
        dh = ops.gemm(dyh, wh[l].t(), M=M, N=dims[l], K=dims[l + 1])
        if l == 0:
            assert torch.equal(dx, dh)
            break
        pre, post, _, mean, rstd = sv[l - 1]
        dy, dg, dbeta = ops.layernorm_bwd(dh, post, pre, mean, rstd, gs[l - 1], relu=True)
        dn = torch.where(post > 0, dh, torch.zeros_like(dh))
        xh = (pre - mean[:, None]) * rstd[:, None]
        _sum_close(dbetas[l - 1], dn, M)
        tol = (M + 2) * 2 * U * (dn.double() * xh.double()).abs().sum(0) * 1.01
        assert bool(((dgs[l - 1].double() - (dn.double() * xh.double()).sum(0)).abs() <= tol).all())


@pytest.mark.parametrize("n,H,W", [(1, 3, 3), (3, 5, 4), (2, 9, 16), (37, 15, 15)])
@pytest.mark.parametrize("relu", [False, True])
def test_conv32_layer(n, H, W, relu):
    from paper_2602_21203_gb300 import ops
    x, w, b, dy = _rand(n, 32, H, W, seed=1), _rand(32, 32, 3, 3, seed=2) * 0.06, _rand(32, seed=3), _rand(n, 32, H - 2, W - 2, seed=4)
    xp = ops.to_phwc(x)
    wf, wb = ops.conv32_layouts(w)
    ref = ops.conv32_fwd(xp, H, W, wf, b, relu)[1]
    _dirty()
    y, xs, wbs = ops.conv32_layer_fwd(x, w, b, relu)
    assert torch.equal(y, ref) and torch.equal(xs, xp) and torch.equal(wbs, wb)
    dyp = ops.to_phwc(ops.relu_bwd(dy, y) if relu else dy)
    _dirty()
    dx, dw, db = ops.conv32_layer_bwd(dy, y if relu else None, xs, wbs)
    assert torch.equal(dx, ops.conv32_dgrad(dyp, H - 2, W - 2, wb)[1])
    rw, rb = ops.wgrad32(xp, dyp, H, W)
    assert torch.equal(dw, rw) and torch.equal(db, rb)
    assert ops.conv32_layer_bwd(dy, None, xs, wbs, need_dx=False)[0] is None


@pytest.mark.parametrize("rows,K", [(1, 2), (7, 51), (512, 101), (2049, 200), (5000, 129)])
def test_ce_mean(rows, K):
    from paper_2602_21203_gb300 import ops
    logits, m = 2 * _rand(rows, K, seed=1), torch.softmax(_rand(rows, K, seed=2), 1)
    row_loss, d, _ = ops.categorical_ce(logits, m, -1.0, 1.0, 0.75 / rows)
    _dirty()
    loss = ops.ce_mean(logits, m)
    assert abs(float(loss) - float(row_loss.double().mean())) <= (rows + 1) * U * float(row_loss.double().abs().mean())
    got = ops.ce_mean_bwd(logits, m, torch.full((), 0.75, device="cuda"))
    # the same products with the scale rounded on the device: one more rounding of 0.75 / rows
    assert bool(((got - d).abs() <= 2 * U * d.abs() + 1e-45).all())


# one row block (32 rows) more than a grid's y dimension counts
MANY = 32 * 65535 + 1


def test_linear_bf16_backward_over_many_rows():
    from paper_2602_21203_gb300 import ops
    x, w, dy = _rand(MANY, 8, seed=1), _rand(9, 8, seed=2), _rand(MANY, 9, seed=3)
    _, xs, ws = ops.linear_bf16_fwd(x, w, None)
    _dirty()
    dx, dw, db = ops.linear_bf16_bwd(dy, xs, ws)
    dyh = ops.cast_bf16(dy)
    assert torch.equal(dx, ops.gemm(dyh, ws.t(), M=MANY, N=8, K=9))
    assert torch.equal(dw, ops.gemm(dyh.t(), xs.t(), M=9, N=8, K=MANY))
    _sum_close(db, dy, MANY)


def test_mlp_head_backward_over_many_rows():
    test_mlp_head_layer(MANY, 8, 32, 1, 3)


def test_ce_mean_of_losses_whose_sum_overflows():
    from paper_2602_21203_gb300 import ops
    rows = 600
    logits, m = torch.zeros(rows, 3, device="cuda"), torch.zeros(rows, 3, device="cuda")
    logits[:, 1], m[:, 1] = -3e36, 1.0      # every row's loss is 3e36 + log 2
    assert abs(float(ops.ce_mean(logits, m)) / 3e36 - 1) <= (rows + 4) * U


# on both sides of two images a CTA
@pytest.mark.parametrize("n", [607, 609, 1300])
def test_conv32_layer_of_many_images(n):
    test_conv32_layer(n, 7, 6, True)


def test_layer_calls_under_capture():
    """Every one-call layer operation captured into a graph gives the bits of the same calls made at once."""
    from paper_2602_21203_gb300 import ops
    x, w, b, dy = _rand(40, 18, seed=1), _rand(13, 18, seed=2), _rand(13, seed=3), _rand(40, 13, seed=4)
    hw = [_rand(64, 18, seed=5), _rand(64, 64, seed=6) / 8, _rand(13, 64, seed=7) / 8]
    hb, hg, ht = [_rand(n, seed=8) for n in (64, 64, 13)], [1 + 0.1 * _rand(64, seed=9)] * 2, [0.1 * _rand(64, seed=10)] * 2
    cx, cw, cb, cd = _rand(3, 32, 7, 9, seed=11), _rand(32, 32, 3, 3, seed=12) * 0.06, _rand(32, seed=13), _rand(3, 32, 5, 7, seed=14)
    m, up = torch.softmax(_rand(40, 13, seed=15), 1), torch.full((), 0.5, device="cuda")

    def calls():
        y, xh, wh = ops.linear_bf16_fwd(x, w, b)
        out, saved = ops.mlp_head_fwd(x, hw, hb, hg, ht)
        cy, xp, wb = ops.conv32_layer_fwd(cx, cw, cb)
        dx, *grads = ops.mlp_head_bwd(dy, hg, saved, 18)
        return [y, *ops.linear_bf16_bwd(dy, xh, wh), *ops.linear_bwd(dy, x, w), out, dx, *[g for gs in grads for g in gs], cy,
                *ops.conv32_layer_bwd(cd, cy, xp, wb), ops.ce_mean(out, m), ops.ce_mean_bwd(out, m, up)]
    want = calls()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        got = calls()
    graph.replay()
    torch.cuda.synchronize()
    assert len(got) == len(want) and all(torch.equal(a, b) for a, b in zip(got, want))
