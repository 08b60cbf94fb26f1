"""Layer operations of include/squint_ops.h on torch CUDA tensors (marshalling only).

Each call launches the library's kernel on the current torch stream.  There is
no fallback: tensors must be CUDA tensors of the stated dtype and layout.
"""
import ctypes

import torch

from . import lib as _lib

DT_F32, DT_F64, DT_BF16 = 0, 1, 2
_DT = {torch.float32: DT_F32, torch.float64: DT_F64, torch.bfloat16: DT_BF16}


def _p(t):
    return None if t is None else t.data_ptr()


def _s():
    """The current stream of the current device as an integer (cudaStream_t)."""
    return torch._C._cuda_getCurrentRawStream(torch.cuda.current_device())


def _chk(rc, what):
    if rc != 0:
        raise _lib.SquintError(rc, what)


def _need(t, dtype, name):
    if not t.is_cuda or t.dtype != dtype:
        raise TypeError(f"{name}: expected a CUDA {dtype} tensor, got {t.dtype} on {t.device}")


def gemm(A, B, bias=None, out=None, accumulate=False, M=None, N=None, K=None):
    """out[m, n] (+)= sum_k A(m, k) B(n, k) + bias; A, B 2-D views given as (rows = m|n, cols = k) with any strides.

    For BF16 operands each of A, B must have one unit stride; out and bias are FP32.
    """
    M = A.shape[0] if M is None else M
    K = A.shape[1] if K is None else K
    N = B.shape[0] if N is None else N
    dt = _DT[A.dtype]
    odt = torch.float32 if dt == DT_BF16 else A.dtype
    if out is None:   # (every element is written unless it is added to)
        out = (torch.zeros if accumulate else torch.empty)(M, N, device=A.device, dtype=odt)
    _need(out, odt, "out")
    if bias is not None:
        _need(bias, odt, "bias")
    _chk(_lib.load().squint_op_gemm(dt, M, N, K, _p(A), A.stride(0), A.stride(1), _p(B), B.stride(0), B.stride(1),
                                    _p(out), out.stride(0), _p(bias), int(accumulate), _s()), "squint_op_gemm")
    return out


def squint_store(frames, ring_obs, slot0, f):
    """Squint at insert: uint8 frames [n, C, H, W] -> rounded f x f means into ring_obs
    [n_slots, C, H/f, W/f] at slots slot0, slot0 + 1, ... (mod n_slots)."""
    _need(frames, torch.uint8, "frames")
    _need(ring_obs, torch.uint8, "ring_obs")
    n, c, h, w = frames.shape
    frames = frames.contiguous()
    _chk(_lib.load().squint_op_squint_store(n, c, h, w, int(f), _p(frames), _p(ring_obs), int(slot0),
                                            ring_obs.shape[0], _s()), "squint_op_squint_store")


def gemm_layernorm(A, B, bias, g, beta, eps=1e-5, relu=True):
    """BF16 A [M, K] B [N, K]^T + bias, then LayerNorm (+ReLU) per row in the same kernel.
    Returns (pre, post, post_bf16, mean, rstd)."""
    _need(A, torch.bfloat16, "A")
    _need(B, torch.bfloat16, "B")
    M, K = A.shape
    N = B.shape[0]
    dev = A.device
    pre = torch.empty(M, N, device=dev)
    post = torch.empty(M, N, device=dev)
    post_bf = torch.empty(M, N, device=dev, dtype=torch.bfloat16)
    mean = torch.empty(M, device=dev)
    rstd = torch.empty(M, device=dev)
    _chk(_lib.load().squint_op_gemm_layernorm(M, N, K, _p(A), A.stride(0), _p(B), B.stride(0), _p(bias), _p(g),
                                              _p(beta), float(eps), int(relu), _p(pre), _p(post), _p(post_bf),
                                              _p(mean), _p(rstd), _s()), "squint_op_gemm_layernorm")
    return pre, post, post_bf, mean, rstd


def cast_bf16(x):
    """FP32 [rows, cols] -> BF16 (round to nearest even) in a buffer whose row stride is
    cols rounded up to 8 (the tensor-core operand alignment); returns the [rows, cols] view."""
    _need(x, torch.float32, "x")
    rows, cols = x.shape
    ld = (cols + 7) // 8 * 8
    buf = torch.empty(rows, ld, dtype=torch.bfloat16, device=x.device)
    if x.stride(1) != 1:
        x = x.contiguous()
    _chk(_lib.load().squint_op_cast_bf16(rows, cols, _p(x), x.stride(0), _p(buf), ld, _s()), "squint_op_cast_bf16")
    return buf[:, :cols]


def mlp_bf16(x, ws, biases, gs, betas, eps=1e-5, save=True, cluster=0):
    """A LayerNorm MLP head in one launch: hidden layers Linear -> LayerNorm -> ReLU
    (weights ws[l] BF16 [out, in], biases FP32), then a plain Linear output layer.
    x BF16 [M, kin].  Returns (out [M, nout], saved) with saved = per hidden layer
    (pre, post, post_bf16, mean, rstd) if save, else None."""
    _need(x, torch.bfloat16, "x")
    nh = len(ws) - 1
    M, kin = x.shape
    H, nout = ws[0].shape[0], ws[-1].shape[0]
    dev = x.device
    for w in ws:
        _need(w, torch.bfloat16, "w")
    out = torch.empty(M, nout, device=dev)

    def arr(ctype, vals):
        return (ctype * len(vals))(*vals)

    P = ctypes.c_void_p
    saved = None
    pre = post = pbf = mean = rstd = None
    if save:
        saved = [(torch.empty(M, H, device=dev), torch.empty(M, H, device=dev),
                  torch.empty(M, H, device=dev, dtype=torch.bfloat16), torch.empty(M, device=dev),
                  torch.empty(M, device=dev)) for _ in range(nh)]
        pre, post, pbf, mean, rstd = (arr(P, [t[i].data_ptr() for t in saved]) for i in range(5))
    _chk(_lib.load().squint_op_mlp_bf16(M, kin, nh, H, nout, _p(x), x.stride(0), arr(P, [w.data_ptr() for w in ws]),
                                        arr(ctypes.c_int64, [w.stride(0) for w in ws]),
                                        arr(P, [b.data_ptr() for b in biases]), arr(P, [g.data_ptr() for g in gs]),
                                        arr(P, [b.data_ptr() for b in betas]), float(eps), _p(out), out.stride(0),
                                        pre, post, pbf, mean, rstd, int(cluster), _s()), "squint_op_mlp_bf16")
    return out, saved


def mlp_bf16_bwd(dout, ws, gs, saved, kin, c0, ncols, want_dpre=True, want_cols=True, betas=None):
    """The input-gradient chain of a head evaluated by mlp_bf16 (saved = its per-layer
    (pre, post, post_bf16, mean, rstd)): dout BF16 [M, nout], weights as for mlp_bf16.
    With betas (the LayerNorm shifts) the ReLU mask is rebuilt from pre and post is not read.
    Returns (dx [M, ncols] = columns c0 .. c0 + ncols of the input gradient,
    dpre_bf16 per hidden layer or None, colpart per hidden layer [ceil(M/128), 3, H] or None)."""
    _need(dout, torch.bfloat16, "dout")
    nh = len(ws) - 1
    M, nout = dout.shape
    H = ws[0].shape[0]
    dev = dout.device
    dx = torch.empty(M, ncols, device=dev)

    def arr(ctype, vals):
        return (ctype * len(vals))(*vals)

    P = ctypes.c_void_p
    dp = [torch.empty(M, H, device=dev, dtype=torch.bfloat16) for _ in range(nh)] if want_dpre else None
    cp = [torch.empty((M + 127) // 128, 3, H, device=dev) for _ in range(nh)] if want_cols else None
    _chk(_lib.load().squint_op_mlp_bwd_bf16(
        M, kin, nh, H, nout, _p(dout), dout.stride(0), arr(P, [w.data_ptr() for w in ws]),
        arr(ctypes.c_int64, [w.stride(0) for w in ws]), arr(P, [t.data_ptr() for t in gs]),
        arr(P, [t.data_ptr() for t in betas]) if betas is not None else None,
        arr(P, [sv[0].data_ptr() for sv in saved]),
        arr(P, [sv[1].data_ptr() for sv in saved]) if betas is None else None,
        arr(P, [sv[3].data_ptr() for sv in saved]), arr(P, [sv[4].data_ptr() for sv in saved]),
        arr(P, [t.data_ptr() for t in dp]) if dp else None, arr(P, [t.data_ptr() for t in cp]) if cp else None,
        int(c0), int(ncols), _p(dx), dx.stride(0), _s()), "squint_op_mlp_bwd_bf16")
    return dx, dp, cp


def gemm_fp8(A, B, bias=None, out=None):
    """out = scale_A scale_B e4m3(A / scale_A) e4m3(B / scale_B)^T + bias for BF16 A [M, K], B [N, K]
    (row-major, unit column stride); per-tensor scales amax / 448.  Returns (out, (scale_A, scale_B))."""
    _need(A, torch.bfloat16, "A")
    _need(B, torch.bfloat16, "B")
    M, K = A.shape
    N = B.shape[0]
    L = _lib.load()
    work = torch.empty(max(L.squint_op_gemm_fp8_workspace(M, N, K), 16), dtype=torch.uint8, device=A.device)
    if out is None:
        out = torch.empty(M, N, device=A.device, dtype=torch.float32)
    if bias is not None:
        _need(bias, torch.float32, "bias")
    _chk(L.squint_op_gemm_fp8(M, N, K, _p(A), A.stride(0), _p(B), B.stride(0), _p(out), out.stride(0), _p(bias),
                              _p(work), work.numel(), _s()), "squint_op_gemm_fp8")
    scales = work[2048:2056].view(torch.float32)
    return out, (scales[0], scales[1])


def quantize_mxfp8(X):
    """MX-FP8 codes and scale bytes of BF16 X [rows, cols] (row-major): returns (codes uint8
    [rows, ceil16(cols)], sf uint8 [squint_op_mx_scale_bytes(rows, cols)])."""
    _need(X, torch.bfloat16, "X")
    rows, cols = X.shape
    L = _lib.load()
    ld8 = (cols + 15) // 16 * 16
    codes = torch.empty(rows, ld8, dtype=torch.uint8, device=X.device)
    sf = torch.empty(max(L.squint_op_mx_scale_bytes(rows, cols), 16), dtype=torch.uint8, device=X.device)
    _chk(L.squint_op_quantize_mxfp8(rows, cols, _p(X), X.stride(0), _p(codes), codes.stride(0), _p(sf), _s()),
         "squint_op_quantize_mxfp8")
    return codes, sf


def gemm_mxfp8(A8, sfa, B8, sfb, K, bias=None, out=None):
    """out = dequant(A) dequant(B)^T + bias for MX-FP8 operands (codes [M, >=K], [N, >=K] with
    their scale bytes from quantize_mxfp8)."""
    M, N = A8.shape[0], B8.shape[0]
    if out is None:
        out = torch.empty(M, N, device=A8.device, dtype=torch.float32)
    if bias is not None:
        _need(bias, torch.float32, "bias")
    _chk(_lib.load().squint_op_gemm_mxfp8(M, N, K, _p(A8), A8.stride(0), _p(sfa), _p(B8), B8.stride(0), _p(sfb),
                                          _p(out), out.stride(0), _p(bias), _s()), "squint_op_gemm_mxfp8")
    return out


def conv3x3_fwd(x, w, b, stride, relu):
    n, cin, h, wd = x.shape
    cout = w.shape[0]
    oh, ow = (h - 3) // stride + 1, (wd - 3) // stride + 1
    y = torch.empty(n, cout, oh, ow, device=x.device, dtype=x.dtype)
    _chk(_lib.load().squint_op_conv3x3_fwd(_DT[x.dtype], n, cin, h, wd, cout, stride, _p(x), _p(w), _p(b), _p(y),
                                           int(relu), _s()), "squint_op_conv3x3_fwd")
    return y


def conv3x3_bwd(x, w, dy, stride, need_dx=True, dx_mask=None):
    n, cin, h, wd = x.shape
    cout = w.shape[0]
    L = _lib.load()
    dt = _DT[x.dtype]
    ws = L.squint_op_conv3x3_workspace(dt, n, cin, h, wd, cout, stride)
    work = torch.empty(max(ws, 16), dtype=torch.uint8, device=x.device)
    dw = torch.empty_like(w)
    db = torch.empty(cout, device=x.device, dtype=x.dtype)
    dx = torch.empty_like(x) if need_dx else None
    _chk(L.squint_op_conv3x3_bwd(dt, n, cin, h, wd, cout, stride, _p(x), _p(w), _p(dy), _p(dx), _p(dx_mask), _p(dw),
                                 _p(db), _p(work), work.numel(), _s()), "squint_op_conv3x3_bwd")
    return dx, dw, db


def relu_bwd(dy, y, out=None):
    """dy * (y > 0) for F32/F64 tensors of the same shape (out may be dy itself)."""
    _need(y, dy.dtype, "y")
    dy, y = dy.contiguous(), y.contiguous()
    out = torch.empty_like(dy) if out is None else out
    _chk(_lib.load().squint_op_relu_bwd(_DT[dy.dtype], dy.numel(), _p(dy), _p(y), _p(out), _s()), "squint_op_relu_bwd")
    return out


def layernorm_fwd(x, g, b, eps=1e-5, relu=False):
    rows, n = x.shape
    y = torch.empty_like(x)
    mean = torch.empty(rows, device=x.device, dtype=torch.float32)
    rstd = torch.empty_like(mean)
    _chk(_lib.load().squint_op_layernorm_fwd(rows, n, _p(x), _p(g), _p(b), float(eps), int(relu), _p(y), _p(mean),
                                             _p(rstd), _s()), "squint_op_layernorm_fwd")
    return y, mean, rstd


def layernorm_bwd(dy, y, x, mean, rstd, g, relu=False):
    rows, n = x.shape
    dx = torch.empty_like(x)
    dg = torch.empty_like(g)
    db = torch.empty_like(g)
    _chk(_lib.load().squint_op_layernorm_bwd(rows, n, _p(dy), _p(y) if relu else None, _p(x), _p(mean), _p(rstd),
                                             _p(g), _p(dx), _p(dg), _p(db), _s()), "squint_op_layernorm_bwd")
    return dx, dg, db


def categorical_ce(logits, m, v_min, v_max, scale):
    rows, K = logits.shape
    d = torch.empty_like(logits)
    loss = torch.empty(rows, device=logits.device, dtype=torch.float32)
    q = torch.empty_like(loss)
    _chk(_lib.load().squint_op_categorical_ce(rows, K, _p(logits), _p(m), float(v_min), float(v_max), float(scale),
                                              _p(d), _p(loss), _p(q), _s()), "squint_op_categorical_ce")
    return loss, d, q


def c51_project(logits, r, d, logp, alpha, gamma, v_min, v_max):
    E, rows, K = logits.shape
    m = torch.empty(rows, K, device=logits.device, dtype=torch.float32)
    _chk(_lib.load().squint_op_c51_project(rows, K, E, _p(logits), _p(r), _p(d), _p(logp), float(alpha), float(gamma),
                                           float(v_min), float(v_max), _p(m), _s()), "squint_op_c51_project")
    return m


def tanh_gaussian_fwd(out, eps, lo=-5.0, hi=2.0):
    rows, A = eps.shape
    a = torch.empty_like(eps)
    logp = torch.empty(rows, device=out.device, dtype=torch.float32)
    _chk(_lib.load().squint_op_tanh_gaussian_fwd(rows, A, _p(out), _p(eps), float(lo), float(hi), _p(a), _p(logp),
                                                 _s()), "squint_op_tanh_gaussian_fwd")
    return a, logp


def tanh_gaussian_bwd(out, eps, da, dlogp, lo=-5.0, hi=2.0):
    rows, A = eps.shape
    dout = torch.empty_like(out)
    _chk(_lib.load().squint_op_tanh_gaussian_bwd(rows, A, _p(out), _p(eps), _p(da), _p(dlogp), float(lo), float(hi),
                                                 _p(dout), _s()), "squint_op_tanh_gaussian_bwd")
    return dout


# ---------------------------------------------------------------- layers, one call a direction
def _ptrs(tensors):
    return (ctypes.c_void_p * len(tensors))(*[t.data_ptr() for t in tensors])


def _addrs(base, step, n):
    return (ctypes.c_void_p * n)(*[base + i * step for i in range(n)])


def _pad8(n):
    return (n + 7) // 8 * 8


def linear_bf16_fwd(x, w, b):
    """bf16(x) bf16(w)^T + b for FP32 x [rows, n_in], w [n_out, n_in].  Returns (y, xh, wh): the BF16
    operands for the backward, row strides rounded up to 8."""
    _need(x, torch.float32, "x")
    _need(w, torch.float32, "w")
    if b is not None:
        _need(b, torch.float32, "bias")
    M, K = x.shape
    N = w.shape[0]
    if x.stride(1) != 1:
        x = x.contiguous()
    if w.stride(1) != 1:
        w = w.contiguous()
    ld = _pad8(K)
    xh, wh = x.new_empty((M, ld), dtype=torch.bfloat16), x.new_empty((N, ld), dtype=torch.bfloat16)
    y = x.new_empty((M, N))
    _chk(_lib.load().squint_op_linear_bf16_fwd(M, N, K, x.data_ptr(), x.stride(0), w.data_ptr(), w.stride(0), _p(b),
                                               xh.data_ptr(), ld, wh.data_ptr(), ld, y.data_ptr(), _s()),
         "squint_op_linear_bf16_fwd")
    return y, xh[:, :K], wh[:, :K]


def linear_bf16_bwd(dy, xh, wh, need=(True, True, True)):
    """(dx, dw, db) of linear_bf16_fwd from dy [rows, n_out] FP32 (contiguous); None where not needed."""
    _need(dy, torch.float32, "dy")
    L = _lib.load()
    M, N = dy.shape
    K = xh.shape[1]
    dx = dy.new_empty((M, K)) if need[0] else None
    dw = dy.new_empty((N, K)) if need[1] else None
    db = dy.new_empty(N) if need[2] else None
    ld = _pad8(N)
    wb = L.squint_op_linear_bf16_bwd_workspace(M, N) if need[2] else 0
    buf = dy.new_empty(M * ld * 2 + wb, dtype=torch.uint8)      # bf16(dy), then the workspace
    _chk(L.squint_op_linear_bf16_bwd(M, N, K, dy.data_ptr(), xh.data_ptr(), xh.stride(0), wh.data_ptr(), wh.stride(0),
                                     buf.data_ptr(), ld, _p(dx), _p(dw), _p(db), buf.data_ptr() + M * ld * 2, wb, _s()),
         "squint_op_linear_bf16_bwd")
    return dx, dw, db


def linear_bwd(dy, x, w, need=(True, True, True)):
    """(dx, dw, db) of the FP32 y = x w^T + b from dy [rows, n_out] (contiguous); None where not needed."""
    _need(dy, torch.float32, "dy")
    M, N = dy.shape
    K = x.shape[1]
    dx = dy.new_empty((M, K)) if need[0] else None
    dw = dy.new_empty((N, K)) if need[1] else None
    db = dy.new_empty(N) if need[2] else None
    _chk(_lib.load().squint_op_linear_bwd(M, N, K, dy.data_ptr(), x.data_ptr(), x.stride(0), x.stride(1), w.data_ptr(),
                                          w.stride(0), w.stride(1), _p(dx), _p(dw), _p(db), _s()), "squint_op_linear_bwd")
    return dx, dw, db


def mlp_head_fwd(x, ws, biases, gs, betas, eps=1e-5):
    """A LayerNorm MLP head from FP32 x [M, kin] and FP32 weights.  Returns (out, saved): saved =
    (xh, wh, pre, post, post_bf, stats) with the BF16 weights in one buffer, the hidden layers'
    pre-activations and outputs as [layers, M, H] and their (mean, rstd) as [2, layers, M]."""
    _need(x, torch.float32, "x")
    nh = len(ws) - 1
    if x.stride(1) != 1:
        x = x.contiguous()
    ws = [w if w.stride(1) == 1 else w.contiguous() for w in ws]
    for w in ws:
        _need(w, torch.float32, "w")
    M, kin = x.shape
    H, nout = ws[0].shape[0], ws[-1].shape[0]
    lds = [_pad8(w.shape[1]) for w in ws]
    xh = x.new_empty((M, _pad8(kin)), dtype=torch.bfloat16)
    sizes = [w.shape[0] * ld for w, ld in zip(ws, lds)]
    wh = x.new_empty(sum(sizes), dtype=torch.bfloat16)
    out = x.new_empty((M, nout))
    pre, post = x.new_empty((nh, M, H)), x.new_empty((nh, M, H))
    post_bf = x.new_empty((nh, M, H), dtype=torch.bfloat16)
    stats = x.new_empty((2, nh, M))
    at, wp = wh.data_ptr(), []
    for n in sizes:
        wp.append(at)
        at += 2 * n
    P, I64 = ctypes.c_void_p, ctypes.c_int64
    _chk(_lib.load().squint_op_mlp_head_fwd(
        M, kin, nh, H, nout, x.data_ptr(), x.stride(0), _ptrs(ws), (I64 * (nh + 1))(*[w.stride(0) for w in ws]),
        _ptrs(biases), _ptrs(gs), _ptrs(betas), float(eps), xh.data_ptr(), xh.stride(0), (P * (nh + 1))(*wp),
        (I64 * (nh + 1))(*lds), out.data_ptr(), _addrs(pre.data_ptr(), 4 * M * H, nh), _addrs(post.data_ptr(), 4 * M * H, nh),
        _addrs(post_bf.data_ptr(), 2 * M * H, nh), _addrs(stats.data_ptr(), 4 * M, nh),
        _addrs(stats.data_ptr() + 4 * nh * M, 4 * M, nh), _s()), "squint_op_mlp_head_fwd")
    return out, (xh, wh, pre, post, post_bf, stats)


def mlp_head_bwd(dout, gs, saved, kin):
    """Gradients of mlp_head_fwd from dout [M, nout] (contiguous): (dx, dws, dbs, dgs, dbetas)."""
    _need(dout, torch.float32, "dout")
    xh, wh, pre, post, post_bf, stats = saved
    L = _lib.load()
    nh, M, H = pre.shape
    nout = dout.shape[1]
    ins = [kin] + [H] * nh
    outs = [H] * nh + [nout]
    lds = [_pad8(k) for k in ins]
    at, wp = wh.data_ptr(), []
    for n, ld in zip(outs, lds):
        wp.append(at)
        at += 2 * n * ld
    dx = dout.new_empty((M, kin))
    dws = [dout.new_empty((n, k)) for n, k in zip(outs, ins)]
    dbs = [dout.new_empty(n) for n in outs]
    dgs = [dout.new_empty(H) for _ in range(nh)]
    dbetas = [dout.new_empty(H) for _ in range(nh)]
    wb = L.squint_op_mlp_head_bwd_workspace(M, nh, H, nout)
    work = dout.new_empty(max(wb, 1), dtype=torch.uint8)
    P, I64 = ctypes.c_void_p, ctypes.c_int64
    _chk(L.squint_op_mlp_head_bwd(
        M, kin, nh, H, nout, dout.data_ptr(), xh.data_ptr(), xh.stride(0), (P * (nh + 1))(*wp), (I64 * (nh + 1))(*lds),
        _ptrs(gs), _addrs(pre.data_ptr(), 4 * M * H, nh), _addrs(post.data_ptr(), 4 * M * H, nh),
        _addrs(post_bf.data_ptr(), 2 * M * H, nh), _addrs(stats.data_ptr(), 4 * M, nh),
        _addrs(stats.data_ptr() + 4 * nh * M, 4 * M, nh), dx.data_ptr(), _ptrs(dws), _ptrs(dbs), _ptrs(dgs), _ptrs(dbetas),
        work.data_ptr(), wb, _s()), "squint_op_mlp_head_bwd")
    return dx, dws, dbs, dgs, dbetas


def conv32_layer_fwd(x, w, b, relu=True):
    """The 32 -> 32 channel convolution layer from NCHW FP32 x.  Returns (y, xp, w_bwd): the padded-HWC
    BF16 input and the data gradient's filter layout for the backward."""
    n, c, H, W = x.shape
    assert c == 32 and x.dtype == torch.float32
    _need(x, torch.float32, "x")
    xp = x.new_empty((n, (H + 4) * (W + 4), 32), dtype=torch.bfloat16)
    wl = x.new_empty((2, 9 * 32 * 32), dtype=torch.bfloat16)
    y = x.new_empty((n, 32, H - 2, W - 2))
    w = w.contiguous()
    _chk(_lib.load().squint_op_conv32_layer_fwd(n, H, W, x.data_ptr(), w.data_ptr(), b.data_ptr(), int(relu), xp.data_ptr(),
                                                wl.data_ptr(), wl.data_ptr() + 9 * 32 * 32 * 2, y.data_ptr(), _s()),
         "squint_op_conv32_layer_fwd")
    return y, xp, wl[1]


def conv32_layer_bwd(dy, y, xp, w_bwd, need_dx=True):
    """(dx, dw, db) of conv32_layer_fwd from dy [n, 32, H-2, W-2] (contiguous); y: the ReLU's output, or None."""
    n, _, oh, ow = dy.shape
    H, W = oh + 2, ow + 2
    L = _lib.load()
    dx = dy.new_empty((n, 32, H, W)) if need_dx else None
    dw, db = dy.new_empty((32, 32, 3, 3)), dy.new_empty(32)
    pb = n * (oh + 4) * (ow + 4) * 64
    wb = max(L.squint_op_wgrad32_workspace(n), 16)
    buf = dy.new_empty(pb + wb, dtype=torch.uint8)      # bf16(dy) padded HWC, then the workspace
    _chk(L.squint_op_conv32_layer_bwd(n, H, W, dy.data_ptr(), _p(y), xp.data_ptr(), w_bwd.data_ptr(), buf.data_ptr(), _p(dx),
                                      dw.data_ptr(), db.data_ptr(), buf.data_ptr() + pb, wb, _s()),
         "squint_op_conv32_layer_bwd")
    return dx, dw, db


def ce_mean(logits, m):
    """Mean over rows of -sum_j m[r, j] log softmax(logits[r])_j, a 0-d tensor (nothing waits for it)."""
    _need(logits, torch.float32, "logits")
    _need(m, torch.float32, "m")
    rows, K = logits.shape
    buf = logits.new_empty(rows)
    loss = logits.new_empty(())
    _chk(_lib.load().squint_op_ce_mean_fwd(rows, K, logits.data_ptr(), m.data_ptr(), buf.data_ptr(), loss.data_ptr(), _s()),
         "squint_op_ce_mean_fwd")
    return loss


def ce_mean_bwd(logits, m, dloss):
    """Gradient of ce_mean at the logits, times the device scalar dloss."""
    _need(dloss, torch.float32, "dloss")
    rows, K = logits.shape
    d = torch.empty_like(logits)
    _chk(_lib.load().squint_op_ce_mean_bwd(rows, K, logits.data_ptr(), m.data_ptr(), dloss.data_ptr(), d.data_ptr(), _s()),
         "squint_op_ce_mean_bwd")
    return d


# ---------------------------------------------------------------- tensor-core convolutions (32 -> 32, stride 1)
def phwc_empty(nimg, H, W, device="cuda"):
    """A zero-filled padded-HWC BF16 buffer for nimg images of H x W x 32."""
    return torch.zeros(nimg, (H + 4) * (W + 4), 32, dtype=torch.bfloat16, device=device)


def to_phwc(x):
    n, c, H, W = x.shape
    assert c == 32 and x.dtype == torch.float32
    out = phwc_empty(n, H, W, x.device)
    _chk(_lib.load().squint_op_to_phwc(n, H, W, _p(x.contiguous()), _p(out), _s()), "squint_op_to_phwc")
    return out


def from_phwc(t, H, W):
    n = t.shape[0]
    out = torch.empty(n, 32, H, W, device=t.device, dtype=torch.float32)
    _chk(_lib.load().squint_op_from_phwc(n, H, W, _p(t), _p(out), _s()), "squint_op_from_phwc")
    return out


def conv0_bf16(x, w, bias, stride, out=None):
    """The encoder's first layer on tensor cores: x NCHW FP32 [n, Cin, H, W], w [32, Cin, 3, 3],
    bias [32] -> ReLU(conv + bias) as padded-HWC BF16 (interior written; `out` defaults to a
    zero-filled buffer)."""
    n, cin, H, W = x.shape
    OH, OW = (H - 3) // stride + 1, (W - 3) // stride + 1
    if out is None:
        out = phwc_empty(n, OH, OW, x.device)
    _chk(_lib.load().squint_op_conv0_bf16(n, cin, H, W, int(stride), _p(x.contiguous()), _p(w.contiguous()),
                                          _p(bias.contiguous()), _p(out), _s()), "squint_op_conv0_bf16")
    return out


def conv32_layouts(w):
    fwd = torch.empty(9 * 32 * 32, dtype=torch.bfloat16, device=w.device)
    bwd = torch.empty_like(fwd)
    _chk(_lib.load().squint_op_conv32_layouts(_p(w.contiguous()), _p(fwd), _p(bwd), _s()), "squint_op_conv32_layouts")
    return fwd, bwd


def conv32_fwd(x_phwc, H, W, w_fwd, bias, relu=True):
    n = x_phwc.shape[0]
    y = phwc_empty(n, H - 2, W - 2, x_phwc.device)
    y_nchw = torch.empty(n, 32, H - 2, W - 2, device=x_phwc.device)
    _chk(_lib.load().squint_op_conv32(0, n, H, W, _p(x_phwc), _p(w_fwd), _p(bias), int(relu), None, _p(y), _p(y_nchw),
                                      _s()), "squint_op_conv32")
    return y, y_nchw


def conv32_dgrad(dy_phwc, H, W, w_bwd, mask_phwc=None):
    n = dy_phwc.shape[0]
    dx = phwc_empty(n, H + 2, W + 2, dy_phwc.device)
    dx_nchw = torch.empty(n, 32, H + 2, W + 2, device=dy_phwc.device)
    _chk(_lib.load().squint_op_conv32(1, n, H, W, _p(dy_phwc), _p(w_bwd), None, 0, _p(mask_phwc), _p(dx),
                                      _p(dx_nchw), _s()), "squint_op_conv32")
    return dx, dx_nchw


def wgrad32(x_phwc, dy_phwc, H, W):
    n = x_phwc.shape[0]
    L = _lib.load()
    work = torch.empty(max(L.squint_op_wgrad32_workspace(n), 16), dtype=torch.uint8, device=x_phwc.device)
    dw = torch.empty(32, 32, 3, 3, device=x_phwc.device)
    db = torch.empty(32, device=x_phwc.device)
    _chk(L.squint_op_wgrad32(n, H, W, _p(x_phwc), _p(dy_phwc), _p(dw), _p(db), _p(work), work.numel(), _s()),
         "squint_op_wgrad32")
    return dw, db
