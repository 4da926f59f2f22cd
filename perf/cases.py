"""The MoE layer's performance cases: the calls a serving program makes, at
the sizes this repository's configurations, tests and benchmark use.

A case names a configuration of ``configs.py`` (its shape, gating and data
type), the call and the tokens of each micro-batch.  ``listed`` holds the
standing cases, ``draw`` makes more of the same ranges, ``prepare`` builds what
a serving program holds before the call (handle, workspace, hidden states),
``run`` makes one call, ``work`` counts the bytes and operations the call
cannot do without, and ``exact`` gives its outputs in float64.

Calls:
  layer     asap_moe_layer on one micro-batch
  batched   asap_moe_layer_batched on micro-batches that are ready together
  mailbox   one post per DP-group stream, served in one round on the MoE stream
  route, dispatch, combine
            the single steps on one micro-batch
The single steps do not read the expert matrices; their handles carry the
narrow FFN of the routing configuration.
"""
import math

import numpy as np
import torch

from paper_2606_22541_gb300 import api
from paper_2606_22541_gb300.configs import CONFIGS

DEV = "cuda"
BLK = 128  # rows, columns and channels of an FP8 scale block


def listed():
    return [
        # the smallest layer of the test suite: launches and latency
        dict(name="layer_tiny_96", call="layer", config="tiny", tokens="96"),
        # a few wide experts, an ordinary micro-batch of that workload
        dict(name="layer_mixtral_1536", call="layer", config="mixtral", tokens="1536"),
        # the benchmark's micro-batch: 256 experts, balanced routing, 128 rows per expert
        dict(name="layer_dsv3_4096", call="layer", config="dsv3_bf16", tokens="4096"),
        # skewed expert popularity, the shortest and the longest prompt batch of that workload
        dict(name="layer_stress_362", call="layer", config="dsv3_stress", tokens="362"),
        dict(name="layer_stress_8045", call="layer", config="dsv3_stress", tokens="8045"),
        # e4m3 experts: a short ragged micro-batch, and the workload's own
        dict(name="layer_fp8_1108", call="layer", config="dsv3_fp8", tokens="1108"),
        dict(name="layer_fp8_4096", call="layer", config="dsv3_fp8", tokens="4096"),
        # four DP groups' micro-batches ready together: the tensor-bound regime
        dict(name="batched_dsv3_4x4096", call="batched", config="dsv3_bf16", tokens="4096,4096,4096,4096"),
        # ragged posts of four DP groups through the mailbox, e4m3 experts
        dict(name="mailbox_fp8_4", call="mailbox", config="dsv3_fp8", tokens="4014,1179,2591,362"),
        # the layer's steps on their own (the token metadata, the payload, the return path)
        dict(name="route_dsv3_4096", call="route", config="dsv3_routing_profile", tokens="4096"),
        dict(name="dispatch_dsv3_2591", call="dispatch", config="dsv3_routing_profile", tokens="2591"),
        dict(name="combine_dsv3_4096", call="combine", config="dsv3_routing_profile", tokens="4096"),
    ]


def _log_uniform(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    call, config, lo, hi, count = rng.choice([
        ("layer", "tiny", 1, 512, 1),
        ("layer", "mixtral", 64, 8192, 1),
        ("layer", "dsv3_bf16", 64, 8192, 1),
        ("layer", "dsv3_stress", 64, 8192, 1),
        ("layer", "dsv3_fp8", 64, 8192, 1),
        ("batched", "dsv3_bf16", 128, 4096, rng.randint(2, 4)),
        ("mailbox", "dsv3_fp8", 128, 4096, rng.randint(2, 4)),
        ("route", "dsv3_routing_profile", 1, 16384, 1),
        ("dispatch", "dsv3_routing_profile", 16, 8192, 1),
        ("combine", "dsv3_routing_profile", 16, 8192, 1),
    ])
    tokens = ",".join(str(_log_uniform(rng, lo, hi)) for _ in range(count))
    return dict(call=call, config=config, tokens=tokens)


def _tokens(case):
    return [int(t) for t in case["tokens"].split(",")]


# ------------------------------------------------------------------ inputs

def _randn(shape, std, seed, stream):
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + stream)
    return torch.randn(shape, generator=g, device=DEV, dtype=torch.float32).mul_(std)


def _zipf_bias(cfg, seed):
    """Router column 0 of the skewed workloads: expert shares follow r^-s."""
    lp = -cfg.zipf_s * np.log(np.arange(1, cfg.n_experts + 1, dtype=np.float64))
    b = lp[np.random.Generator(np.random.PCG64(seed)).permutation(cfg.n_experts)]
    return torch.tensor(cfg.zipf_beta * (b - b.mean()), dtype=torch.float32, device=DEV)


def _hidden_states(cfg, n, seed, i):
    x = _randn((n, cfg.hidden), 1.0, seed, 100 + i).to(torch.bfloat16)
    if cfg.zipf_s is not None:
        x[:, 0] = 1.0
    return x


def _router(cfg, seed):
    wr = _randn((cfg.n_experts, cfg.hidden), 0.02 if cfg.name == "tiny" else cfg.hidden ** -0.5, seed, 1)
    if cfg.zipf_s is not None:
        wr[:, 0] = _zipf_bias(cfg, seed)
    return wr.to(torch.bfloat16)


def _block_e4m3(w):
    """fp32 [R, C] as e4m3 with one scale amax / 448 per 128 x 128 block."""
    R, C = w.shape
    b = w.view(R // BLK, BLK, C // BLK, BLK)
    amax = b.abs().amax(dim=(1, 3))
    s = torch.where(amax > 0, amax / 448.0, torch.ones_like(amax))
    return (b / s[:, None, :, None]).clamp_(-448.0, 448.0).to(torch.float8_e4m3fn).view(R, C), s


def _matrix(cfg, rows, cols, seed, stream):
    """One expert matrix [rows, cols] (N(0, 1/cols)) as stored: (values, scales or None)."""
    w = _randn((rows, cols), cols ** -0.5, seed, stream)
    return (w.to(torch.bfloat16), None) if cfg.dtype == "bf16" else _block_e4m3(w)


# matrix kind -> (stream of the generator, rows and columns of a configuration)
_KINDS = {"gate": (1000, lambda c, i: (i, c.hidden)), "up": (2000, lambda c, i: (i, c.hidden)),
          "down": (3000, lambda c, i: (c.hidden, i))}


def _expert(cfg, kind, e, seed):
    stream, shape = _KINDS[kind]
    return _matrix(cfg, *shape(cfg, cfg.inter), seed, stream + e)


def _shared(cfg, kind, seed):
    stream, shape = _KINDS[kind]
    return _matrix(cfg, *shape(cfg, cfg.shared_inter), seed, stream + 900)


def _weights(cfg, seed):
    w = dict(router_w=_router(cfg, seed), router_bias=None)
    dt = torch.bfloat16 if cfg.dtype == "bf16" else torch.float8_e4m3fn
    for kind, (_, shape) in _KINDS.items():
        r, c = shape(cfg, cfg.inter)
        stack = torch.empty((cfg.n_experts, r, c), dtype=dt, device=DEV)
        scales = torch.empty((cfg.n_experts, r // BLK, c // BLK), device=DEV) if cfg.dtype != "bf16" else None
        for e in range(cfg.n_experts):
            v, s = _expert(cfg, kind, e, seed)
            stack[e] = v
            if s is not None:
                scales[e] = s
        w["w_" + kind], w["s_" + kind] = stack, scales
        if cfg.n_shared:
            w["sh_" + kind], w["sh_s_" + kind] = _shared(cfg, kind, seed)
    return w


def _combine_inputs(cfg, n, seed):
    """Expert outputs, shared rows, weights and a permutation as the steps before leave them."""
    nk = n * cfg.top_k
    y = _randn((nk, cfg.hidden), 0.5, seed, 200).to(torch.bfloat16)
    ysh = _randn((n, cfg.hidden), 0.5, seed, 201).to(torch.bfloat16)
    w = _randn((n, cfg.top_k), 1.0, seed, 202).sigmoid_()
    w = (w / w.sum(1, keepdim=True) * cfg.route_scale).contiguous()
    g = torch.Generator(device=DEV)
    g.manual_seed(int(seed) * 1009 + 203)
    pd = torch.randperm(nk, generator=g, device=DEV).to(torch.int32).view(n, cfg.top_k)
    return y, ysh, w, pd


def _dispatch_idx(cfg, n, seed):
    """k different experts per token, as routing leaves them."""
    s = _randn((n, cfg.n_experts), 1.0, seed, 204)
    return s.topk(cfg.top_k, dim=1).indices.to(torch.int32).contiguous()


# ------------------------------------------------------------------ the calls

def prepare(case, seed):
    cfg, ns, call = CONFIGS[case["config"]], _tokens(case), case["call"]
    total = sum(ns)
    h = api.asap_moe_create(cfg, _weights(cfg, seed), total)
    st = dict(call=call, h=h, ns=ns)
    if call == "combine":
        st["y"], st["ysh"], st["w"], st["pd"] = _combine_inputs(cfg, total, seed)
        st["out"] = torch.empty((total, cfg.hidden), dtype=torch.bfloat16, device=DEV)
        return st
    st["x"] = [_hidden_states(cfg, n, seed, i) for i, n in enumerate(ns)]
    if call == "mailbox":
        st["box"] = api.asap_moe_mailbox_create(h, len(ns), max(ns))
        st["streams"] = [torch.cuda.Stream() for _ in ns]
        st["moe"] = torch.cuda.Stream()
    else:
        st["ws"] = api.workspace(h, total)
    i32 = dict(dtype=torch.int32, device=DEV)
    nk = total * cfg.top_k
    if call == "route":
        st["idx"] = torch.empty((total, cfg.top_k), **i32)
        st["w"] = torch.empty((total, cfg.top_k), device=DEV)
        st["counts"], st["offsets"] = torch.empty(cfg.n_experts, **i32), torch.empty(cfg.n_experts + 1, **i32)
    elif call == "dispatch":
        st["idx"] = _dispatch_idx(cfg, total, seed)
        st["xp"] = torch.empty((nk, cfg.hidden), dtype=torch.bfloat16, device=DEV)
        st["ps"], st["pd"] = torch.empty(nk, **i32), torch.empty((total, cfg.top_k), **i32)
    else:
        st["out"] = [torch.empty_like(x) for x in st["x"]]
    return st


def run(st):
    call, h = st["call"], st["h"]
    if call == "layer":
        api.asap_moe_layer(h, st["x"][0], st["out"][0], st["ws"])
        return st["out"][0]
    if call == "batched":
        api.asap_moe_layer_batched(h, st["x"], st["out"], st["ws"])
        return st["out"]
    if call == "mailbox":
        cur = torch.cuda.current_stream()
        slots = list(range(len(st["x"])))
        epochs = []
        for i in slots:
            st["streams"][i].wait_stream(cur)  # the group's hidden states are ready
            epochs.append(api.asap_moe_mailbox_post(st["box"], i, st["x"][i], st["out"][i], stream=st["streams"][i]))
        api.asap_moe_mailbox_serve_many(st["box"], slots, epochs, stream=st["moe"])
        for i in slots:
            api.asap_moe_mailbox_wait(st["box"], i, stream=cur)
        return st["out"]
    if call == "route":
        api.asap_moe_route(h, st["x"][0], st["idx"], st["w"], st["counts"], st["offsets"], st["ws"])
        return [st["idx"], st["w"], st["counts"], st["offsets"]]
    if call == "dispatch":
        api.asap_moe_dispatch(h, st["x"][0], st["idx"], st["xp"], st["ps"], st["pd"], st["ws"])
        return [st["xp"], st["ps"], st["pd"]]
    api.asap_moe_combine(h, st["y"], st["ysh"], st["w"], st["pd"], st["out"])
    return st["out"]


# Tail of the skewed workloads' token shares.  It is steeper than zipf_s (the
# fit to ranks 2..64): 191, 223 and 244 experts have rows at 256, 512 and 1024
# tokens on a GB300; exponent 1.3 gives 179, 220 and 246.
_ZIPF_TAIL = 1.3


def _active_experts(cfg, n):
    """Expected number of experts with at least one row among n tokens."""
    E = cfg.n_experts
    p = np.ones(E) if cfg.zipf_s is None else np.arange(1, E + 1, dtype=np.float64) ** -_ZIPF_TAIL
    p = np.minimum(p / p.sum() * cfg.top_k, 1.0)
    return float((1.0 - (1.0 - p) ** n).sum())


def work(case):
    cfg, ns, call = CONFIGS[case["config"]], _tokens(case), case["call"]
    n, H, k, E = sum(ns), cfg.hidden, cfg.top_k, cfg.n_experts
    row = 2 * H  # bytes of a bf16 token row
    if call == "route":
        return dict(bytes=n * row + E * row + n * k * 8 + (2 * E + 1) * 4, flops=2 * n * H * E)
    if call == "dispatch":
        return dict(bytes=n * row + n * k * row + n * k * 12, flops=0)
    if call == "combine":
        return dict(bytes=n * k * (row + 8) + 2 * n * row, flops=2 * n * (k + 1) * H)
    # the whole layer: hidden states in, outputs out, every active expert's weights once
    wb = 2.0 if cfg.dtype == "bf16" else 1.0 + 4.0 / (BLK * BLK)
    weights = 3 * H * wb * (_active_experts(cfg, n) * cfg.inter + cfg.n_shared * cfg.shared_inter)
    return dict(bytes=int(2 * n * row + E * row + weights),
                flops=n * (cfg.flops_per_token() + cfg.router_flops_per_token()))


# ------------------------------------------------------------------ float64

def _route64(cfg, x, wr):
    logits = x.double() @ wr.double().t()
    n, E, k = logits.shape[0], cfg.n_experts, cfg.top_k
    if cfg.gating == "sigmoid_grouped":
        s = logits.sigmoid()
        grp = s.view(n, cfg.n_groups, -1)
        kept = grp.topk(2, dim=2).values.sum(2).topk(cfg.topk_groups, dim=1).indices
        mask = torch.zeros((n, cfg.n_groups), dtype=torch.bool, device=DEV).scatter_(1, kept, True)
        sel = torch.where(mask[:, :, None].expand_as(grp).reshape(n, E), s, torch.full_like(s, -1.0))
        idx = sel.topk(k, dim=1).indices
        w = s.gather(1, idx)
        return idx, w / w.sum(1, keepdim=True) * cfg.route_scale
    idx = logits.topk(k, dim=1).indices
    p = logits.softmax(1) if cfg.gating == "softmax" else None
    return idx, p.gather(1, idx) if p is not None else logits.gather(1, idx).softmax(1)


def _decode(v, s):
    if s is None:
        return v.double()
    R, C = v.shape
    return (v.float().double().view(R // BLK, BLK, C // BLK, BLK) * s.double()[:, None, :, None]).view(R, C)


def _quantised(cfg, a):
    """a as an FP8 expert matrix meets it: e4m3 per row per 128 channels."""
    if cfg.dtype == "bf16":
        return a
    b = a.view(a.shape[0], -1, BLK)
    amax = b.abs().amax(dim=2, keepdim=True)
    s = torch.where(amax > 0, amax / 448.0, torch.ones_like(amax))
    q = (b / s).clamp(-448.0, 448.0).float().to(torch.float8_e4m3fn)
    return (q.float().double() * s).view_as(a)


def _swiglu64(cfg, xq, gate, up, down):
    g = xq @ _decode(*gate).t()
    h = torch.nn.functional.silu(g) * (xq @ _decode(*up).t())
    return _quantised(cfg, h) @ _decode(*down).t()


def _layer64(cfg, x, seed):
    idx, w = _route64(cfg, x, _router(cfg, seed))
    xq = _quantised(cfg, x.double())
    kinds = ("gate", "up", "down")
    out = torch.zeros_like(xq)
    for e in range(cfg.n_experts):
        t, j = (idx == e).nonzero(as_tuple=True)
        if t.numel():
            y = _swiglu64(cfg, xq[t], *(_expert(cfg, kind, e, seed) for kind in kinds))
            out.index_add_(0, t, y * w[t, j][:, None])
    if cfg.n_shared:
        out += _swiglu64(cfg, xq, *(_shared(cfg, kind, seed) for kind in kinds))
    return out


def exact(case, seed):
    cfg, ns, call = CONFIGS[case["config"]], _tokens(case), case["call"]
    if call == "dispatch":
        return None  # copies and whole numbers
    if call == "combine":
        y, ysh, w, pd = _combine_inputs(cfg, sum(ns), seed)
        out = ysh.double()
        for j in range(cfg.top_k):
            out += w[:, j:j + 1].double() * y[pd[:, j].long()].double()
        return out
    xs = [_hidden_states(cfg, n, seed, i) for i, n in enumerate(ns)]
    if call == "route":
        return [None, _route64(cfg, xs[0], _router(cfg, seed))[1], None, None]
    if work(case)["flops"] > 1.6e13:
        return None  # over 20 s in float64
    out = _layer64(cfg, torch.cat(xs), seed)
    return out if call == "layer" else list(out.split(ns))
