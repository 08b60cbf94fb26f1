"""The policy head and the categorical target over action and atom counts, against FP64."""
import pytest
import torch

pytestmark = pytest.mark.gpu

U = 2.0 ** -24


# actions a row around the 8, 16 and 32 threads that share it; rows that do not fill a block
@pytest.mark.parametrize("A", [1, 6, 8, 9, 16, 17, 32, 33, 70])
@pytest.mark.parametrize("rows", [1, 19, 512])
def test_tanh_gaussian(rows, A):
    from paper_2602_21203_gb300 import ops
    g = torch.Generator().manual_seed(100 * A + rows)
    out, eps = torch.randn(rows, 2 * A, generator=g).cuda(), torch.randn(rows, A, generator=g).cuda()
    a, logp = ops.tanh_gaussian_fwd(out, eps)
    o, e = out.double(), eps.double()
    mu, raw = o[:, :A], o[:, A:]
    ls = -5.0 + 3.5 * (torch.tanh(raw) + 1)
    u = mu + ls.exp() * e
    sp = torch.nn.functional.softplus(-2 * u)
    assert float((a.double() - torch.tanh(u)).abs().max()) <= 64 * U * float(1 + (ls.exp() * e).abs().max())
    term = -0.5 * e * e - ls - 0.91893853320467274 - 2 * (0.69314718055994531 - u - sp)
    # some 20 operations a term, on values of the size of its parts (u moves by its own size times that of the
    # log scale's error); then one addition an action
    size = 0.5 * e * e + ls.abs() + 1 + 2 * (0.7 + (1 + 7) * (mu.abs() + (ls.exp() * e).abs()) + sp)
    tol = 32 * U * size.sum(1) + A * U * term.abs().sum(1)
    assert bool(((logp.double() - term.sum(1)).abs() <= tol).all())
    da, dl = torch.randn(rows, A, generator=g).cuda(), torch.randn(rows, generator=g).cuda()
    mu2, raw2 = mu.clone().requires_grad_(), raw.clone().requires_grad_()
    u2 = mu2 + (-5.0 + 3.5 * (torch.tanh(raw2) + 1)).exp() * e
    l2 = (-0.5 * e * e - (-5.0 + 3.5 * (torch.tanh(raw2) + 1)) - 2 * (0.69314718055994531 - u2 -
          torch.nn.functional.softplus(-2 * u2))).sum(1)
    ((torch.tanh(u2) * da.double()).sum() + (l2 * dl.double()).sum()).backward()
    dout = ops.tanh_gaussian_bwd(out, eps, da, dl)
    ref = torch.cat([mu2.grad, raw2.grad], 1)
    scale = (1 + da.double().abs().max() + dl.double().abs().max()) * (1 + 3.5 * 2) * float(1 + (ls.exp() * e).abs().max()) ** 2
    assert float((dout.double() - ref).abs().max()) <= 64 * U * float(scale)


@pytest.mark.parametrize("K", [2, 31, 33, 101, 128, 129, 256])
@pytest.mark.parametrize("rows,E", [(1, 1), (7, 2), (130, 3)])
def test_categorical_target(rows, E, K):
    from paper_2602_21203_gb300 import ops
    g = torch.Generator().manual_seed(10 * K + rows + E)
    lg, r = torch.randn(E, rows, K, generator=g).cuda(), torch.randn(rows, generator=g).cuda()
    d, lp = (torch.rand(rows, generator=g) < 0.3).float().cuda(), torch.randn(rows, generator=g).cuda()
    m = ops.c51_project(lg, r, d, lp, 0.1, 0.97, -4.0, 6.0)
    z = torch.linspace(-4.0, 6.0, K, dtype=torch.float64, device="cuda")
    p = torch.softmax(lg.double(), 2).mean(0)
    alpha, gamma = torch.tensor(0.1).double().item(), torch.tensor(0.97).double().item()
    tz = (r.double()[:, None] + gamma * (1 - d.double()[:, None]) * (z - alpha * lp.double()[:, None])).clamp(-4.0, 6.0)
    b = ((tz + 4.0) / (10.0 / (K - 1))).clamp(0, K - 1)
    w = (1 - (b[:, :, None] - torch.arange(K, device="cuda")).abs()).clamp(min=0)
    want = (p[:, :, None] * w).sum(1)
    # an atom's place errs by some 8 roundings of a number up to K - 1 + |z| / dz, which moves its whole
    # probability by that much; probabilities and the sums add 16 + K roundings
    tol = (8 * (2 * K) * U * 4 + (16 + K) * U) * 1.0
    assert float((m.double() - want).abs().max()) <= tol
    assert float((m.double().sum(1) - 1).abs().max()) <= K * tol


# both ends of every count of atoms a lane
@pytest.mark.parametrize("K", [32, 64, 65, 96, 97, 160, 161, 192, 193, 224, 225])
def test_categorical_target_atoms_a_lane(K):
    test_categorical_target(13, 2, K)
