"""The work this library does for its users, as timed cases.

Every case calls a public entry point (``paper_2609_23733_gb300.binding``) the way a program
does: inputs, weights, workspace and output buffers exist on the GPU before the call, and one
pass is one call (``vp_linear``, ``vp_router``, ``vp_head_attention``, one routed layer, one
block of the stack, the stack).  Model shapes are VGGT's global aggregator (D = 1024, 16 heads
of 64, FFN ratio 4); token counts are views times tokens per view (261 at 224 px, 1,374 at
518 px), so every listed size is ragged against 128-row tiles.

``exact`` evaluates the same formulas in float64 with plain torch, without storage roundings.
"""
from __future__ import annotations

import math

import torch

import paper_2609_23733_gb300.binding as vpb

D_HEAD = 64
MEAN, SURROGATE, FULL = 0, 1, 2
LN_EPS = 1e-6
P224, P518 = 261, 1374  # tokens of a view: 5 special + (px / 14)^2 patches
# Cost of the most expensive drawn case, in the units of _cost (the block at 100 views).
MAX_COST = 8.2e12


def listed():
    return [
        # QKV projection of the smallest workload (4 views at 224 px): a launch-bound GEMM with
        # fewer tiles than SMs.
        {"name": "linear_qkv_s4", "op": "linear", "M": 4 * P224, "K": 1024, "Nout": 3072, "gelu": False,
         "residual": False},
        # FFN up-projection with GELU at 8 views, 518 px: a mid-size GEMM of a few waves.
        {"name": "linear_fc1_s8", "op": "linear", "M": 8 * P518, "K": 1024, "Nout": 4096, "gelu": True,
         "residual": False},
        # FFN down-projection with LayerScale and residual at 32 views: a large GEMM, long K.
        {"name": "linear_fc2_s32", "op": "linear", "M": 32 * P518, "K": 4096, "Nout": 1024, "gelu": False,
         "residual": True},
        # The router on its own, 8 views, with biases and every output (r costs a pass over K):
        # the saliency analyses of a scene.
        {"name": "router_s8", "op": "router", "N": 8 * P518, "H": 16, "bias": True, "all_outputs": True},
        # The router at the largest workload (100 views): two sweeps over Q, K and V.
        {"name": "router_s100", "op": "router", "N": 100 * P518, "H": 16, "bias": False, "all_outputs": False},
        # Every head exact at 8 views, with the MaxAttn saliency: the unrouted attention.
        {"name": "heads_full_s8", "op": "heads", "N": 8 * P518, "H": 16, "full": 16, "surrogate": 0,
         "s_attn": True},
        # A layer without full heads at 64 views (the routing-mix sweep's 0 % point): surrogate
        # and mean heads.
        {"name": "heads_cheap_s64", "op": "heads", "N": 64 * P518, "H": 16, "full": 0, "surrogate": 8,
         "s_attn": False},
        # One routed layer of the smallest workload, a quarter of the heads exact.
        {"name": "layer_s4", "op": "layer", "N": 4 * P224, "H": 16, "full": 4, "surrogate": 6, "rope": False,
         "P": P224, "grid": 16},
        # One routed layer at 32 views with qk-norm and 2-D RoPE, the paper's average mix.
        {"name": "layer_qk_s32", "op": "layer", "N": 32 * P518, "H": 16, "full": 1, "surrogate": 7,
         "rope": True, "P": P518, "grid": 37},
        # One block of the headline stack (100 views), the paper's average mix.
        {"name": "block_s100", "op": "stack", "N": 100 * P518, "H": 16, "layers": 1, "full": 1, "surrogate": 7,
         "merge": 0, "P": P518},
        # The same block with token merging at stride 10 (about 90 % of the tokens merged).
        {"name": "block_merge_s100", "op": "stack", "N": 100 * P518, "H": 16, "layers": 1, "full": 1,
         "surrogate": 7, "merge": 10, "P": P518},
        # The whole 24-block stack at 4 views: many short launches.
        {"name": "stack_s4", "op": "stack", "N": 4 * P224, "H": 16, "layers": 24, "full": 1, "surrogate": 7,
         "merge": 0, "P": P224},
    ]


def _log_uniform(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed kinds, sizes spread over the logarithm of their range."""
    while True:
        case = _draw(rng)
        if _cost(case) <= MAX_COST:
            return case


def _draw(rng):
    op = rng.choice(["linear", "linear", "router", "heads", "layer", "stack", "merge"])
    H = rng.choice([8, 12, 16, 16])
    D = H * D_HEAD
    if op == "linear":
        K, Nout, gelu, residual = rng.choice([(D, 3 * D, False, False), (D, 4 * D, True, False),
                                              (4 * D, D, False, True), (D, D, False, True)])
        return {"op": op, "M": _log_uniform(rng, P224, 100 * P518), "K": K, "Nout": Nout, "gelu": gelu,
                "residual": residual}
    if op == "router":
        return {"op": op, "N": _log_uniform(rng, P224, 100 * P518), "H": H, "bias": rng.random() < 0.5,
                "all_outputs": rng.random() < 0.5}
    full = rng.choice([0, 1, 1, 2, H // 4])
    surrogate = rng.randint(0, H - full)
    if op == "heads":
        if rng.random() < 0.25:
            full, surrogate = H, 0
        return {"op": op, "N": _log_uniform(rng, P224, 100 * P518), "H": H, "full": full, "surrogate": surrogate,
                "s_attn": rng.random() < 0.5}
    P, grid = rng.choice([(P224, 16), (P518, 37), (734, 27)])
    views = _log_uniform(rng, 2, 100)
    if op == "layer":
        return {"op": op, "N": views * P, "H": H, "full": full, "surrogate": surrogate,
                "rope": rng.random() < 0.5, "P": P, "grid": grid}
    if op == "merge":
        return {"op": "stack", "N": views * P, "H": H, "layers": 1, "full": full, "surrogate": surrogate,
                "merge": rng.choice([4, 10]), "P": P}
    N = views * P
    layers = rng.randint(2, 24) if N <= 8 * P224 else 1
    return {"op": "stack", "N": N, "H": H, "layers": layers, "full": full, "surrogate": surrogate, "merge": 0,
            "P": P}


# ------------------------------------------------------------------ inputs
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _randn(g, *shape):
    return torch.randn(*shape, generator=g, device="cuda")


def _xavier(g, *shape):
    """Xavier-uniform weight [..., fan_out, fan_in] in bf16."""
    bound = math.sqrt(6.0 / (shape[-1] + shape[-2]))
    return ((torch.rand(*shape, generator=g, device="cuda") * 2 - 1) * bound).to(torch.bfloat16)


def _layer_params(g, H, block):
    D, L = H * D_HEAD, 64
    w = {"w_qkv": _xavier(g, 3 * D, D), "b_qkv": 0.05 * _randn(g, 3 * D),
         "w_o": _xavier(g, D, D), "b_o": 0.05 * _randn(g, D)}
    w.update(_router_params(g, H, False))
    w.update(_surrogate_params(g, H))
    if block:
        for n in ("ln1", "ln2"):
            w[n + "_g"] = 1.0 + 0.1 * _randn(g, D)
            w[n + "_b"] = 0.05 * _randn(g, D)
        w["ls1"] = 1.0 + 0.1 * _randn(g, D)
        w["ls2"] = 1.0 + 0.1 * _randn(g, D)
        w["w_fc1"], w["b_fc1"] = _xavier(g, 4 * D, D), 0.05 * _randn(g, 4 * D)
        w["w_fc2"], w["b_fc2"] = _xavier(g, D, 4 * D), 0.05 * _randn(g, D)
    return w


def _router_params(g, H, bias):
    w = {"r_W": _xavier(g, H, 64, D_HEAD), "r_U": _xavier(g, H, 64, D_HEAD),
         "r_w": _xavier(g, H, 64, 1).reshape(H, 64).contiguous()}
    if bias:
        w["r_bW"], w["r_bU"] = 0.05 * _randn(g, H, 64), 0.05 * _randn(g, H, 64)
    return w


def _surrogate_params(g, H):
    w = {}
    for m in ("g", "d"):
        w[f"s_{m}1_w"], w[f"s_{m}1_b"] = _xavier(g, H, 64, 2 * D_HEAD), 0.05 * _randn(g, H, 64)
        w[f"s_{m}2_w"], w[f"s_{m}2_b"] = _xavier(g, H, D_HEAD, 64), 0.05 * _randn(g, H, D_HEAD)
    return w


def _qk_params(g):
    return {k: (1.0 + 0.1 * _randn(g, 64)) if k.endswith("g") else 0.05 * _randn(g, 64)
            for k in ("q_norm_g", "q_norm_b", "k_norm_g", "k_norm_b")}


def _modes(case, layer=0):
    """Routed modes of a layer: the full heads, then mean and surrogate heads, at rotating
    positions, so that every head slot sees each mode somewhere in a stack."""
    H, full, surr = case["H"], case["full"], case["surrogate"]
    order = [FULL] * full + [MEAN] * (H - full - surr) + [SURROGATE] * surr
    m = [0] * H
    for k in range(H):
        m[(5 * layer + k) % H] = order[k]
    return m


def _salient_qkv(g, N, H):
    """Queries around a per-head direction and keys of which one answers it, so that a third of
    the heads each have a dominant key (full band), a leading one (surrogate band), and none."""
    qkv = torch.randn(N, 3, H, D_HEAD, generator=g, device="cuda", dtype=torch.bfloat16)
    mu = _randn(g, H, D_HEAD)
    qkv[:, 0] = (0.7 * qkv[:, 0].float() + mu).to(torch.bfloat16)
    at = torch.randint(0, N, (H,), generator=g, device="cuda")
    target = torch.tensor([0.0, 0.045, 0.5], device="cuda")[torch.arange(H, device="cuda") % 3]
    var = (0.125 ** 2) * (mu * mu).sum(-1)
    gain = torch.log(target / (1 - target)) + math.log(N) + 0.5 * var
    key = (gain * 8.0 / (mu * mu).sum(-1)).unsqueeze(-1) * mu
    h = torch.arange(H, device="cuda")
    own = qkv[at, 1, h]
    qkv[at, 1, h] = torch.where((target > 0).unsqueeze(-1), key, own.float()).to(torch.bfloat16)
    return qkv


class _State:
    pass


def prepare(case, seed):
    g = _gen(seed)
    st = _State()
    st.case = case
    op = case["op"]
    if op == "linear":
        M, K, Nout = case["M"], case["K"], case["Nout"]
        st.A = torch.randn(M, K, generator=g, device="cuda", dtype=torch.bfloat16)
        st.W, st.bias = _xavier(g, Nout, K), 0.05 * _randn(g, Nout)
        st.scale = 1.0 + 0.1 * _randn(g, Nout) if case["residual"] else None
        st.res = torch.randn(M, Nout, generator=g, device="cuda", dtype=torch.bfloat16) if case["residual"] else None
        st.act = vpb.VP_ACT_GELU if case["gelu"] else vpb.VP_ACT_NONE
        return st
    N, H = case["N"], case["H"]
    st.dm = vpb.dims(N, H)
    if op == "router":
        st.qkv = _salient_qkv(g, N, H)
        st.w = _router_params(g, H, case["bias"])
        st.rw = vpb.router_weights(st.w)
        st.s = torch.zeros(H, device="cuda")
        st.modes = torch.zeros(H, dtype=torch.int32, device="cuda")
        more = case["all_outputs"]
        st.q_pool, st.ctx, st.mean_v = (torch.zeros(H, D_HEAD, device="cuda") for _ in range(3))
        st.r = torch.zeros(H, N, device="cuda") if more else None
        st.ws = vpb.workspace(st.dm, vpb.VP_WS_ROUTER)
        return st
    if op == "heads":
        st.qkv = torch.randn(N, 3, H, D_HEAD, generator=g, device="cuda", dtype=torch.bfloat16)
        st.w = _surrogate_params(g, H)
        st.sw = vpb.surrogate_weights(st.w)
        modes = torch.tensor(_modes(case), dtype=torch.int32)
        st.head_ids = torch.argsort(modes, stable=True).to(torch.int32).cuda()
        counts = [0] + [int((modes == m).sum()) for m in range(3)]
        st.offsets = torch.tensor(counts).cumsum(0).to(torch.int32).cuda()
        st.mean_v = st.qkv[:, 2].float().mean(0).contiguous()
        st.ctx = (st.mean_v + 0.5 * _randn(g, H, D_HEAD)).contiguous()
        st.y = torch.empty(N, H * D_HEAD, dtype=torch.bfloat16, device="cuda")
        st.s_attn = torch.zeros(H, device="cuda") if case["s_attn"] else None
        st.ws = vpb.workspace(st.dm, vpb.VP_WS_ROUTER)
        return st
    D = H * D_HEAD
    st.x0 = torch.randn(N, D, generator=g, device="cuda", dtype=torch.bfloat16)
    if op == "layer":
        st.w = _layer_params(g, H, False)
        st.rw, st.sw = vpb.router_weights(st.w), vpb.surrogate_weights(st.w)
        st.qkw = _qk_params(g) if case["rope"] else None
        st.qk = vpb.qk_options(st.qkw, LN_EPS, True, case["P"], 5, case["grid"], 100.0) if case["rope"] else None
        st.force = torch.tensor(_modes(case), dtype=torch.int32, device="cuda")
        st.out = torch.empty_like(st.x0)
        st.modes = torch.zeros(H, dtype=torch.int32, device="cuda")
        st.ws = vpb.workspace(st.dm, vpb.VP_WS_LAYER)
        return st
    layers = case["layers"]
    st.w = [_layer_params(g, H, True) for _ in range(layers)]
    st.layers = [vpb.layer_weights(w, merge=vpb.merge_options(case["merge"], case["P"]) if case["merge"] else None)
                 for w in st.w]
    st.force = torch.tensor([_modes(case, l) for l in range(layers)], dtype=torch.int32, device="cuda")
    st.x = torch.empty_like(st.x0)
    st.modes = torch.zeros(layers, H, dtype=torch.int32, device="cuda")
    st.ws = vpb.workspace(st.dm, vpb.VP_WS_STACK_MERGE if case["merge"] else vpb.VP_WS_STACK)
    return st


def run(st):
    op = st.case["op"]
    if op == "linear":
        return vpb.vp_linear(st.A, st.W, st.bias, st.act, st.scale, st.res)
    if op == "router":
        vpb.vp_router(st.dm, st.qkv, st.rw, None, st.s, st.modes, st.q_pool, st.ctx, st.mean_v, st.r, st.ws)
        out = {"s": st.s, "modes": st.modes, "q_pool": st.q_pool, "ctx": st.ctx, "mean_v": st.mean_v}
        if st.r is not None:
            out["r"] = st.r
        return out
    if op == "heads":
        vpb.vp_head_attention(st.dm, st.qkv, st.head_ids, st.offsets, st.ctx, st.mean_v, st.sw, st.y, st.ws,
                              s_attn=st.s_attn)
        return {"y": st.y, "s_attn": st.s_attn} if st.s_attn is not None else {"y": st.y}
    if op == "layer":
        w = st.w
        vpb.vp_moh_global_attention(st.dm, st.x0, w["w_qkv"], w["b_qkv"], w["w_o"], w["b_o"], st.rw, st.sw,
                                    st.force, st.out, None, None, None, st.modes, st.ws, qk=st.qk)
        return {"out": st.out, "modes": st.modes}
    st.x.copy_(st.x0)  # the stack works in place: the tokens of this pass
    vpb.vp_global_stack(st.dm, st.x, st.layers, st.force, st.modes, None, LN_EPS, st.ws)
    return {"x": st.x, "modes": st.modes}


# ------------------------------------------------------------------ unavoidable work
def _router_flops(N, H):
    return N * H * (2 * D_HEAD * 128 + 2 * D_HEAD * 4)


def _heads_flops(N, full, surrogate):
    return full * 4.0 * N * N * D_HEAD + surrogate * N * 2.0 * (64 * 128 + 2 * 64 * 64)


def _cost(case):
    """Flops of a case, with a floor for the memory it moves."""
    w = work(case)
    return max(w["flops"], w["bytes"] * 100.0)


def work(case):
    op = case["op"]
    if op == "linear":
        M, K, Nout = case["M"], case["K"], case["Nout"]
        extra = M * Nout * 2 + Nout * 4 if case["residual"] else 0
        return {"bytes": 2 * (M * K + Nout * K + M * Nout) + 4 * Nout + extra, "flops": 2.0 * M * K * Nout}
    N, H = case["N"], case["H"]
    D = H * D_HEAD
    if op == "router":
        return {"bytes": N * 3 * D * 2 + (N * H * 4 if case["all_outputs"] else 0) + H * 64 * 64 * 4,
                "flops": _router_flops(N, H)}
    full, surr = case["full"], case["surrogate"]
    if op == "heads":
        return {"bytes": N * D_HEAD * 2 * (3 * full + surr + H), "flops": _heads_flops(N, full, surr)}
    weights = 2 * (4 * D * D + H * (2 * 64 * 64 + 2 * (64 * 128 + 64 * 64)))
    if op == "layer":
        fl = 2.0 * N * D * 3 * D + _router_flops(N, H) + _heads_flops(N, full, surr) + \
            2.0 * N * (full + surr) * D_HEAD * D
        return {"bytes": 2 * 2 * N * D + weights, "flops": fl}
    layers, stride = case["layers"], case["merge"]
    Np, match = N, 0.0
    if stride:
        P, views = case["P"], N // case["P"]
        Np = P + (views - 1) * (5 + -(-(P - 5) // stride))
        match = 2.0 * N * D * 64 + 2.0 * (N - Np) * Np * D_HEAD
    fl = 2.0 * Np * D * 3 * D + _router_flops(Np, H) + _heads_flops(Np, full, surr) + \
        2.0 * Np * (full + surr) * D_HEAD * D + 2.0 * 2 * N * D * 4 * D + match
    return {"bytes": 2 * 2 * N * D + layers * (weights + 2 * 8 * D * D), "flops": layers * fl}


# ------------------------------------------------------------------ the same in 64 bits
def exact(case, seed):
    if case.get("merge"):
        return None  # the matching is a discrete choice: no value to be near to
    if work(case)["flops"] > 4.0e12:
        return None  # over 20 s in double precision
    st = prepare(case, seed)
    op = case["op"]
    if op == "linear":
        out = st.A.double() @ st.W.double().T + st.bias.double()
        if case["gelu"]:
            out = torch.nn.functional.gelu(out)
        return out * st.scale.double() + st.res.double() if case["residual"] else out
    if op == "router":
        r = _router64(st.qkv, st.w)
        out = {"s": r["s"], "modes": None, "q_pool": r["q_pool"], "ctx": r["ctx"], "mean_v": r["mean_v"]}
        if st.r is not None:
            out["r"] = r["r"]
        return out
    if op == "heads":
        y, s_attn = _heads64(st.qkv, _modes(case), st.ctx.double(), st.mean_v.double(), st.w)
        return {"y": y.flatten(1), "s_attn": s_attn} if case["s_attn"] else {"y": y.flatten(1)}
    if op == "layer":
        rope = (case["P"], 5, case["grid"]) if case["rope"] else None
        return {"out": _attention64(st.x0.double(), st.w, _modes(case), st.qkw, rope), "modes": None}
    x = st.x0.double()
    for l, w in enumerate(st.w):
        x = x + w["ls1"].double() * _attention64(_ln64(x, w["ln1_g"], w["ln1_b"]), w, _modes(case, l), None, None)
        h = torch.nn.functional.gelu(_ln64(x, w["ln2_g"], w["ln2_b"]) @ w["w_fc1"].double().T + w["b_fc1"].double())
        x = x + w["ls2"].double() * (h @ w["w_fc2"].double().T + w["b_fc2"].double())
    return {"x": x, "modes": None}


def _ln64(x, g, b):
    return torch.nn.functional.layer_norm(x, x.shape[-1:], g.double(), b.double(), LN_EPS)


def _router64(qkv, w):
    N, _, H, _ = qkv.shape
    out = {k: [] for k in ("s", "q_pool", "ctx", "mean_v", "r")}
    for h in range(H):
        q, k, v = (qkv[:, i, h].double() for i in range(3))
        a, b = q @ w["r_W"][h].double().T, q @ w["r_U"][h].double().T
        if "r_bW" in w:
            a, b = a + w["r_bW"][h].double(), b + w["r_bU"][h].double()
        alpha = torch.softmax((torch.tanh(a) * torch.sigmoid(b)) @ w["r_w"][h].double(), 0)
        q_pool = alpha @ q
        r = torch.softmax(0.125 * (k @ q_pool), 0)
        for name, val in (("s", r.max()), ("q_pool", q_pool), ("ctx", r @ v), ("mean_v", v.mean(0)), ("r", r)):
            out[name].append(val)
    return {k: torch.stack(v) for k, v in out.items()}


def _heads64(qkv, modes, ctx, mean_v, w):
    N, _, H, d = qkv.shape
    y = torch.zeros(N, H, d, dtype=torch.float64, device=qkv.device)
    s_attn = torch.zeros(H, dtype=torch.float64, device=qkv.device)
    for h in range(H):
        q, k, v = (qkv[:, i, h].double() for i in range(3))
        if modes[h] == FULL:
            for a in range(0, N, 2048):
                p = torch.softmax(0.125 * (q[a:a + 2048] @ k.T), 1)
                y[a:a + 2048, h] = p @ v
                s_attn[h] = torch.maximum(s_attn[h], p.max())
        elif modes[h] == SURROGATE:
            z = torch.cat([v, ctx[h].expand(N, d)], 1)
            g, dl = (torch.nn.functional.gelu(z @ w[f"s_{m}1_w"][h].double().T + w[f"s_{m}1_b"][h].double())
                     @ w[f"s_{m}2_w"][h].double().T + w[f"s_{m}2_b"][h].double() for m in ("g", "d"))
            y[:, h] = ctx[h] + torch.sigmoid(g) * dl
        else:
            y[:, h] = mean_v[h]
    return y, s_attn


def _attention64(x, w, modes, qkw, rope):
    """Routed attention up to W_O: QKV (qk-norm, 2-D RoPE), router, heads, W_O."""
    N, D = x.shape
    H = D // D_HEAD
    qkv = (x @ w["w_qkv"].double().T + w["b_qkv"].double()).reshape(N, 3, H, D_HEAD)
    if qkw is not None:
        for i, t in enumerate(("q", "k")):
            qkv[:, i] = _rope64(_ln64(qkv[:, i], qkw[t + "_norm_g"], qkw[t + "_norm_b"]), *rope)
    r = _router64(qkv, w)
    y, _ = _heads64(qkv, modes, r["ctx"], r["mean_v"], w)
    return y.flatten(1) @ w["w_o"].double().T + w["b_o"].double()


def _rope64(x, P, start, grid):
    """Channels [0, 32) turn with the patch row, [32, 64) with the column, base 100."""
    t = torch.arange(x.shape[0], device=x.device) % P - start
    pos = torch.stack([torch.where(t >= 0, t // grid + 1, 0), torch.where(t >= 0, t % grid + 1, 0)])
    theta = 100.0 ** (-torch.arange(16, dtype=torch.float64, device=x.device) / 16)
    out = x.clone()
    for axis in range(2):
        ang = pos[axis].double()[:, None, None] * theta
        a, b = x[..., 32 * axis:32 * axis + 16], x[..., 32 * axis + 16:32 * axis + 32]
        out[..., 32 * axis:32 * axis + 16] = a * torch.cos(ang) - b * torch.sin(ang)
        out[..., 32 * axis + 16:32 * axis + 32] = b * torch.cos(ang) + a * torch.sin(ang)
    return out
