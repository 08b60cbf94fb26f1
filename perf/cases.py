"""The work that users of this framework have it do, as measurable cases.

Whole calls: training segments (UTD updates as one graph, then the weights read back) and
batched actor inference.  Layers and blocks through `autograd` and `ops`: the encoder's
convolutions, the projections, a LayerNorm MLP head, the losses of one update, and squint
at insert.  Sizes are those of the workloads in paper_2602_21203_gb300/synth.py, the tests
and bench.py; draws spread over the ranges around them, odd sizes among them.
"""
import math
import random

import torch
import torch.nn.functional as F

from paper_2602_21203_gb300 import autograd as ag
from paper_2602_21203_gb300 import lib, ops, synth

_PREC = {"fp32": lib.PREC_FP32, "bf16": lib.PREC_BF16}


def listed():
    return [
        # The training loop of the headline workload: four UTD-4 calls in BF16, then the
        # weights read back (a checkpoint, or actors elsewhere).
        {"name": "update_train_bf16", "kind": "update", "preset": "train_b512", "precision": "bf16", "batch": 512,
         "ring": 100_000, "k": 4, "calls": 4},
        # The same update in FP32, the learner's default precision.
        {"name": "update_train_fp32", "kind": "update", "preset": "train_b512", "precision": "fp32", "batch": 512,
         "ring": 100_000, "k": 4, "calls": 1},
        # The small visual workload: batch 32, one update a call, launches and latency count.
        {"name": "update_small_fp32", "kind": "update", "preset": "small_b32", "precision": "fp32", "batch": 32,
         "ring": 256, "k": 1, "calls": 8},
        # A policy on a few robots (deployment): eight rows, one request.
        {"name": "act_8", "kind": "act", "preset": "train_b512", "precision": "bf16", "rows": 8, "groups": 1},
        # Inference for 4,096 parallel environments in 16 ragged groups.
        {"name": "act_4096", "kind": "act", "preset": "train_b512", "precision": "bf16", "rows": 4096, "groups": 16},
        # The critic head of the training shape, forward and backward.
        {"name": "mlp_head_512", "kind": "mlp_head", "rows": 512, "kin": 274, "hidden": 512, "layers": 2, "out": 101},
        # An inner encoder layer over both frames of a batch of 512 in BF16, forward and backward.
        {"name": "conv32_bf16_1024", "kind": "conv32", "n": 1024, "h": 15, "w": 15},
        # The same layer over one frame in FP32.
        {"name": "conv3x3_fp32_512", "kind": "conv3x3", "n": 512, "cin": 32, "cout": 32, "h": 15, "w": 15, "stride": 1},
        # The projection of the flattened encoder features over a large batch, forward and backward, BF16.
        {"name": "linear_bf16_4096", "kind": "linear", "precision": "bf16", "rows": 4096, "kin": 2592, "out": 256},
        # A hidden layer of the small workload's heads in FP32: a short call.
        {"name": "linear_fp32_32", "kind": "linear", "precision": "fp32", "rows": 32, "kin": 418, "out": 256},
        # Policy sample, projected target, cross entropy and their gradients for one batch.
        {"name": "losses_512", "kind": "losses", "rows": 512, "atoms": 101, "actions": 6},
        # 4,096 rendered frames squinted into the replay ring.
        {"name": "squint_store_4096", "kind": "squint_store", "n": 4096, "h": 128, "w": 128, "f": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["update", "update", "act", "act", "mlp_head", "conv32", "conv3x3", "linear", "linear", "losses",
                       "squint_store"])
    if kind == "update":
        preset = rng.choice(["train_b512", "stored_b512", "state_b512", "small_b32"])
        k = rng.choice([1, 2, 4])
        return {"kind": kind, "preset": preset, "precision": rng.choice(["fp32", "bf16"]), "batch": _log(rng, 16, 512),
                "ring": _log(rng, 1000, 50_000), "k": k, "calls": rng.randint(1, 4) if k < 4 else 1}
    if kind == "act":
        preset = rng.choice(["train_b512", "train_b512", "stored_b512", "state_b512", "small_b32"])
        rows = _log(rng, 1, 4096)
        return {"kind": kind, "preset": preset, "precision": rng.choice(["bf16", "bf16", "fp32"]), "rows": rows,
                "groups": rng.randint(1, min(16, rows))}
    if kind == "mlp_head":
        return {"kind": kind, "rows": _log(rng, 32, 4096), "kin": _log(rng, 18, 512), "hidden": rng.choice([256, 512]),
                "layers": rng.choice([1, 2, 2, 3]), "out": rng.choice([12, 51, 101, rng.randint(1, 128)])}
    if kind == "conv32":
        return {"kind": kind, "n": _log(rng, 8, 2048), "h": rng.randint(7, 17), "w": rng.randint(7, 17)}
    if kind == "conv3x3":
        cin, stride = rng.choice([(3, 2), (16, 1), (32, 1), (32, 2)])
        return {"kind": kind, "n": _log(rng, 8, 512), "cin": cin, "cout": rng.choice([16, 32]), "h": rng.randint(9, 33),
                "w": rng.randint(9, 33), "stride": stride}
    if kind == "linear":
        return {"kind": kind, "precision": rng.choice(["bf16", "fp32"]), "rows": _log(rng, 8, 4096),
                "kin": _log(rng, 18, 2592), "out": _log(rng, 12, 512)}
    if kind == "losses":
        return {"kind": kind, "rows": _log(rng, 32, 8192), "atoms": rng.randint(11, 201), "actions": rng.randint(1, 12)}
    f = rng.choice([1, 2, 4])
    return {"kind": kind, "n": _log(rng, 16, 4096), "h": f * rng.randint(16, 128 // f), "w": f * rng.randint(16, 128 // f),
            "f": f}


# ---------------------------------------------------------------- inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _uniform(g, bound, *shape):
    return (torch.rand(*shape, generator=g, device="cuda") * 2 - 1) * bound


def _config(case):
    over = {k: case[k] for k in ("batch",) if k in case}
    if "ring" in case:
        over["ring_size"] = case["ring"]
    return synth.make_config(case["preset"], **over)


def _conv_sizes(cfg):
    """(cin, cout, h, w, stride, oh, ow) of every encoder layer."""
    out, cin = [], cfg["obs_c"]
    if cfg["conv_layers"] == 0:
        return out
    h, w = cfg["obs_h"] // cfg["squint_f"], cfg["obs_w"] // cfg["squint_f"]
    for layer in range(cfg["conv_layers"]):
        s = 2 if layer == 0 else 1
        oh, ow = (h - 3) // s + 1, (w - 3) // s + 1
        out.append((cin, cfg["conv_ch"], h, w, s, oh, ow))
        cin, h, w = cfg["conv_ch"], oh, ow
    return out


def _shapes(cfg):
    """The flat parameter layout: (name, shape, fan_in) in order."""
    out, convs = [], _conv_sizes(cfg)
    feat = convs[-1][1] * convs[-1][5] * convs[-1][6] if convs else 0
    for i, (ci, co, *_) in enumerate(convs):
        out += [("conv%d.w" % i, (co, ci, 3, 3), ci * 9), ("conv%d.b" % i, (co,), ci * 9)]

    def norm(name, n):
        return [(name + ".g", (n,), 0), (name + ".beta", (n,), 0)]

    def linear(name, n, k):
        return [(name + ".w", (n, k), k), (name + ".b", (n,), k)]

    def mlp(name, k, n_out):
        got = []
        for i, h in enumerate(cfg["hidden"]):
            got += linear("%s%d" % (name, i), h, k) + norm("%s%d" % (name, i), h)
            k = h
        return got + linear(name + "_out", n_out, k)

    z = cfg["proj_dim"] or feat
    proj = cfg["proj_dim"]
    if proj:
        out += linear("cproj", proj, feat) + norm("cproj", proj)
    for e in range(cfg["n_critics"]):
        out += mlp("critic%d_" % e, z + cfg["proprio_dim"] + cfg["action_dim"], cfg["atoms"])
    if proj:
        out += linear("aproj", proj, feat) + norm("aproj", proj)
    out += mlp("actor", z + cfg["proprio_dim"], 2 * cfg["action_dim"])
    return out + [("log_alpha", (1,), 0)]


def _weights(cfg, seed):
    g, got = _gen(seed), {}
    for name, shape, fan in _shapes(cfg):
        if fan:
            got[name] = _uniform(g, fan ** -0.5, *shape)
        elif name.endswith(".g"):
            got[name] = 1 + 0.1 * _randn(g, *shape)
        elif name.endswith(".beta"):
            got[name] = 0.1 * _randn(g, *shape)
        else:
            got[name] = torch.full(shape, math.log(cfg["init_alpha"]), device="cuda")
    return got


def _group_sizes(case):
    """`rows` split into `groups` ragged requests."""
    rows, n = case["rows"], case["groups"]
    cuts = sorted(random.Random(rows * 31 + n).sample(range(1, rows), n - 1)) if n > 1 else []
    return [b - a for a, b in zip([0] + cuts, cuts + [rows])]


def _layer_inputs(case, seed):
    """Tensors of a layer case by name; those under "grad" are differentiated, "dy" is the output's gradient."""
    g, kind = _gen(seed), case["kind"]
    if kind == "mlp_head":
        x = _randn(g, case["rows"], case["kin"])
        params, k = [], case["kin"]
        for _ in range(case["layers"]):
            h = case["hidden"]
            params += [_uniform(g, k ** -0.5, h, k), _uniform(g, k ** -0.5, h), 1 + 0.1 * _randn(g, h), 0.1 * _randn(g, h)]
            k = h
        params += [_uniform(g, k ** -0.5, case["out"], k), _uniform(g, k ** -0.5, case["out"])]
        return [x] + params, _randn(g, case["rows"], case["out"]) / case["rows"]
    if kind == "linear":
        b = case["kin"] ** -0.5
        return [_randn(g, case["rows"], case["kin"]), _uniform(g, b, case["out"], case["kin"]),
                _uniform(g, b, case["out"])], _randn(g, case["rows"], case["out"]) / case["rows"]
    if kind == "conv32":
        cin, cout, s = 32, 32, 1
    else:
        cin, cout, s = case["cin"], case["cout"], case["stride"]
    b = (cin * 9) ** -0.5
    n, h, w = case["n"], case["h"], case["w"]
    return [torch.relu(_randn(g, n, cin, h, w)), _uniform(g, b, cout, cin, 3, 3), _uniform(g, b, cout)], \
        _randn(g, n, cout, (h - 3) // s + 1, (w - 3) // s + 1) / n


def _loss_inputs(case, seed):
    g, B, K, A = _gen(seed), case["rows"], case["atoms"], case["actions"]
    return {"out": _randn(g, B, 2 * A), "eps": _randn(g, B, A), "target": _randn(g, 2, B, K), "logits": _randn(g, B, K),
            "r": _randn(g, B), "d": (torch.rand(B, generator=g, device="cuda") < 0.02).float(),
            "da": _randn(g, B, A) / B, "dlogp": torch.full((B,), 0.1 / B, device="cuda")}


_V, _ALPHA, _GAMMA = 20.0, 0.1, 0.99


def prepare(case, seed):
    kind = case["kind"]
    if kind == "update":
        cfg = _config(case)
        cfg["seed"] = int(seed)
        learner = lib.Learner(cfg, synth.make_ring(cfg, seed, device="cuda"), precision=_PREC[case["precision"]])
        return {"kind": kind, "learner": learner, "k": case["k"], "calls": case["calls"],
                "stats": [lib.PinnedStats(case["k"]) for _ in range(case["calls"])]}
    if kind == "act":
        cfg = _config(case)
        learner = lib.Learner(cfg, None, precision=_PREC[case["precision"]])
        flat = torch.cat([w.reshape(-1) for w in _weights(cfg, seed).values()])
        learner.set_params(flat.cpu().numpy())
        learner.refresh_policy()
        groups = []
        for i, n in enumerate(_group_sizes(case)):
            obs, prop = synth.make_obs_batch(n, cfg, seed * 1000 + i, device="cuda")
            groups.append((obs, prop, torch.empty(n, cfg["action_dim"], device="cuda")))
        reqs = [lib.Learner.request(o, p, a, key=i, sample=False, group_id=i) for i, (o, p, a) in enumerate(groups)]
        return {"kind": kind, "learner": learner, "groups": groups, "requests": reqs}
    if kind == "losses":
        t = _loss_inputs(case, seed)
        t["out"].requires_grad_()
        t["logits"].requires_grad_()
        return {"kind": kind, **t}
    if kind == "squint_store":
        g, n, f = _gen(seed), case["n"], case["f"]
        frames = torch.randint(0, 256, (n, 3, case["h"], case["w"]), dtype=torch.uint8, generator=g, device="cuda")
        ring = torch.zeros(2 * n, 3, case["h"] // f, case["w"] // f, dtype=torch.uint8, device="cuda")
        return {"kind": kind, "frames": frames, "ring": ring, "slot0": 2 * n - n // 2, "f": f}
    ins, dy = _layer_inputs(case, seed)
    return {"kind": kind, "ins": [t.requires_grad_() for t in ins], "dy": dy, "stride": case.get("stride", 1),
            "precision": case.get("precision", "bf16")}


# ---------------------------------------------------------------- one pass
def run(state):
    kind = state["kind"]
    if kind == "update":
        learner = state["learner"]
        for buf in state["stats"]:
            learner.update_async(state["k"], buf)
        weights = learner.params()        # waits for the updates
        rows = [s for buf in state["stats"] for s in buf.read()]
        return {"params": weights, "stats": {k: torch.tensor([s[k] for s in rows]) for k in rows[0]}}
    if kind == "act":
        state["learner"].act(state["requests"])
        return [a for _, _, a in state["groups"]]
    if kind == "losses":
        a, logp = ag.tanh_gaussian(state["out"], state["eps"])
        with torch.no_grad():
            m = ops.c51_project(state["target"], state["r"], state["d"], logp, _ALPHA, _GAMMA, -_V, _V)
        loss = ag.categorical_ce(state["logits"], m, -_V, _V)
        dlogits, = torch.autograd.grad(loss, state["logits"])
        dout, = torch.autograd.grad((a, logp), state["out"], (state["da"], state["dlogp"]))
        return {"a": a, "logp": logp, "m": m, "loss": loss, "dlogits": dlogits, "dout": dout}
    if kind == "squint_store":
        ops.squint_store(state["frames"], state["ring"], state["slot0"], state["f"])
        return state["ring"]
    ins = state["ins"]
    if kind == "mlp_head":
        y = ag.mlp_head_bf16(ins[0], ins[1:])
    elif kind == "conv32":
        y = ag.conv32_bf16(*ins)
    elif kind == "conv3x3":
        y = ag.conv3x3(*ins, state["stride"], True)
    else:
        y = (ag.linear if state["precision"] == "fp32" else ag.linear_bf16)(*ins)
    return [y] + list(torch.autograd.grad(y, ins, state["dy"]))


# ---------------------------------------------------------------- work of one pass
def _head_dims(cfg, critic):
    convs = _conv_sizes(cfg)
    z = cfg["proj_dim"] or (convs[-1][1] * convs[-1][5] * convs[-1][6] if convs else 0)
    k = z + cfg["proprio_dim"] + (cfg["action_dim"] if critic else 0)
    dims = [k] + list(cfg["hidden"]) + [cfg["atoms"] if critic else 2 * cfg["action_dim"]]
    return sum(a * b for a, b in zip(dims, dims[1:])), dims[0] * dims[1]


def _numel(cfg):
    return sum(math.prod(s) for _, s, _ in _shapes(cfg))


def work(case):
    kind = case["kind"]
    if kind in ("update", "act"):
        cfg = _config(case)
        convs = _conv_sizes(cfg)
        conv = [co * ci * 9 * oh * ow for ci, co, _, _, _, oh, ow in convs]
        feat = convs[-1][1] * convs[-1][5] * convs[-1][6] if convs else 0
        proj = feat * cfg["proj_dim"]
        actor, _ = _head_dims(cfg, False)
        frame = cfg["obs_c"] * cfg["obs_h"] * cfg["obs_w"]
        row = frame + 4 * (cfg["proprio_dim"] + cfg["action_dim"])
    if kind == "update":
        B, E, n = cfg["batch"], cfg["n_critics"], _numel(cfg)
        critic, critic0 = _head_dims(cfg, True)
        macs = 2 * sum(conv) + sum(conv) + sum(conv[1:])                       # encoder: both frames; dW, dX on o_t
        macs += 5 * proj + 3 * proj                                            # projections; their dW and the critic's dX
        macs += 2 * actor + 2 * actor                                          # actor on o_t+1, o_t; its backward
        macs += 3 * E * critic + 2 * E * critic + E * critic                   # targets, online, actor step; backwards
        k = case["k"] * case["calls"]
        return {"bytes": k * (2 * B * row + n * 4 * 8) + 4 * n, "flops": 2 * B * macs * k}
    if kind == "act":
        return {"bytes": case["rows"] * row + 4 * _numel(cfg), "flops": 2 * case["rows"] * (sum(conv) + proj + actor)}
    if kind == "mlp_head":
        M, H, n = case["rows"], case["hidden"], case["layers"]
        macs = case["kin"] * H + (n - 1) * H * H + H * case["out"]
        return {"bytes": 4 * (2 * M * case["kin"] + 2 * macs + 2 * M * case["out"]), "flops": 6 * M * macs}
    if kind == "linear":
        M, K, N = case["rows"], case["kin"], case["out"]
        return {"bytes": 4 * (2 * M * K + 2 * N * K + 2 * M * N), "flops": 6 * M * N * K}
    if kind in ("conv32", "conv3x3"):
        ci, co, s = case.get("cin", 32), case.get("cout", 32), case.get("stride", 1)
        oh, ow = (case["h"] - 3) // s + 1, (case["w"] - 3) // s + 1
        return {"bytes": 4 * case["n"] * (2 * ci * case["h"] * case["w"] + 2 * co * oh * ow) + 8 * ci * co * 9,
                "flops": 6 * case["n"] * ci * co * 9 * oh * ow}
    if kind == "losses":
        B, K, A = case["rows"], case["atoms"], case["actions"]
        return {"bytes": 4 * B * (2 * K + K + K + K + 2 * A * 2 + 3 * A + 4), "flops": B * K * (K + 40)}
    px = case["n"] * 3 * case["h"] * case["w"]
    return {"bytes": px + px // case["f"] ** 2, "flops": px}


# ---------------------------------------------------------------- the same in 64 bits
def _conv64(x, w, b, s):
    n, _, h, wd = x.shape
    cols = F.unfold(x, 3, stride=s)
    y = w.reshape(w.shape[0], -1) @ cols + b[:, None]
    return y.reshape(n, w.shape[0], (h - 3) // s + 1, (wd - 3) // s + 1)


def _head64(x, params, eps=1e-5):
    for i in range(0, len(params) - 2, 4):
        w, b, g, beta = params[i:i + 4]
        x = torch.relu(F.layer_norm(x @ w.t() + b, (w.shape[0],), g, beta, eps))
    return x @ params[-2].t() + params[-1]


def _act64(case, seed):
    cfg = _config(case)
    w = {k: v.double() for k, v in _weights(cfg, seed).items()}
    got = []
    for i, n in enumerate(_group_sizes(case)):
        obs, prop = synth.make_obs_batch(n, cfg, seed * 1000 + i, device="cuda")
        x = prop.double()
        if obs is not None:
            z = F.avg_pool2d(obs.double(), cfg["squint_f"]) / 255 - 0.5
            for layer, size in enumerate(_conv_sizes(cfg)):
                z = torch.relu(_conv64(z, w["conv%d.w" % layer], w["conv%d.b" % layer], size[4]))
            z = z.reshape(n, -1)
            if cfg["proj_dim"]:
                z = F.layer_norm(z @ w["aproj.w"].t() + w["aproj.b"], (cfg["proj_dim"],), w["aproj.g"], w["aproj.beta"],
                                 cfg["ln_eps"])
            x = torch.cat([z, x], 1)
        y = _head64(x, [v for k, v in w.items() if k.startswith("actor")], cfg["ln_eps"])
        got.append(torch.tanh(y[:, :cfg["action_dim"]]))
    return got


def _losses64(case, seed):
    t = {k: v.double() for k, v in _loss_inputs(case, seed).items()}
    out, K = t["out"].requires_grad_(), case["atoms"]
    mu, raw = out.chunk(2, 1)
    log_std = -5.0 + 3.5 * (torch.tanh(raw) + 1)
    u = mu + log_std.exp() * t["eps"]
    a = torch.tanh(u)
    logp = (-0.5 * t["eps"] ** 2 - log_std - 0.5 * math.log(2 * math.pi)
            - 2 * (math.log(2.0) - u - F.softplus(-2 * u))).sum(1)
    with torch.no_grad():
        p = torch.softmax(t["target"], 2).mean(0)
        z = torch.linspace(-_V, _V, K, dtype=torch.float64, device="cuda")
        tz = (t["r"][:, None] + _GAMMA * (1 - t["d"])[:, None] * (z - _ALPHA * logp[:, None])).clamp(-_V, _V)
        b = (tz + _V) / (2 * _V / (K - 1))
        m = torch.stack([(p * (1 - (b - j).abs()).clamp(min=0)).sum(1) for j in range(K)], 1)
    logits = t["logits"].requires_grad_()
    loss = -(m * torch.log_softmax(logits, 1)).sum(1).mean()
    dlogits, = torch.autograd.grad(loss, logits)
    dout, = torch.autograd.grad((a, logp), out, (t["da"], t["dlogp"]))
    return {"a": a, "logp": logp, "m": m, "loss": loss, "dlogits": dlogits, "dout": dout}


def exact(case, seed):
    kind = case["kind"]
    if kind in ("update", "squint_store"):
        return None
    if kind == "act":
        return _act64(case, seed)
    if kind == "losses":
        return _losses64(case, seed)
    ins, dy = _layer_inputs(case, seed)
    ins, dy = [t.double().requires_grad_() for t in ins], dy.double()
    if kind == "mlp_head":
        y = _head64(ins[0], ins[1:])
    elif kind == "linear":
        y = ins[0] @ ins[1].t() + ins[2]
    else:
        y = torch.relu(_conv64(*ins, case.get("stride", 1)))
    return [y] + list(torch.autograd.grad(y, ins, dy))
