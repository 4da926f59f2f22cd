"""The histogram and scan of dispatch, by one cluster (up to 8192 tokens) and by
a launch each, over chunk ranges of every kind and one to eight blocks of 32
experts, against a stable sort; the scan of the gate (by the gate's own cluster
up to 256 tokens) against a count and against dispatch."""
import pytest
import torch

from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("experts", [1, 32, 33, 100, 256])
@pytest.mark.parametrize("n", [1, 33, 65, 1025, 8192, 8193, 32769, 66000])
def test_scan(experts, n):
    k = min(2, experts)
    cfg = inputs.small_variant(MIXTRAL, name="scan", hidden=256, inter=256, n_experts=experts, top_k=k, seed=5)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), n)
    g = torch.Generator(device=DEV).manual_seed(n * 1000 + experts)
    # skewed towards the low experts, some unused
    first = (torch.rand(n, generator=g, device=DEV) ** 3 * experts).int().clamp_(max=experts - 1)
    idx = torch.stack([(first + j) % experts for j in range(k)], 1).contiguous()
    x = torch.zeros((n, cfg.hidden), dtype=torch.bfloat16, device=DEV)
    x[:, 0] = torch.arange(n, device=DEV) % 256
    xp = torch.empty((n * k, cfg.hidden), dtype=torch.bfloat16, device=DEV)
    src = torch.empty(n * k, dtype=torch.int32, device=DEV)
    dst = torch.empty((n, k), dtype=torch.int32, device=DEV)
    for _ in range(2):  # the second call finds the first one's workspace
        api.asap_moe_dispatch(h, x, idx, xp, src, dst, api.workspace(h, n))
    order = torch.sort(idx.flatten().long(), stable=True).indices
    assert api.asap_moe_status(h) == (0, 0)
    assert torch.equal(dst.flatten().long()[order], torch.arange(n * k, device=DEV))
    assert torch.equal(src.long(), order // k)
    assert torch.equal(xp, x[order // k])


@pytest.mark.parametrize("experts", [8, 16, 24, 32, 64, 128, 256])
@pytest.mark.parametrize("n", [1, 17, 32, 33, 65, 129, 255, 256, 257])
def test_gate_scan(experts, n):
    cfg = inputs.small_variant(MIXTRAL, name="gate", hidden=256, inter=256, n_experts=experts, top_k=2, seed=6)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), n)
    x = inputs.make_tokens(cfg, n, 0, DEV)
    ws = api.workspace(h, n)
    i32 = dict(dtype=torch.int32, device=DEV)
    idx, w = torch.empty((n, 2), **i32), torch.empty((n, 2), device=DEV)
    counts, offs = torch.empty(experts, **i32), torch.empty(experts + 1, **i32)
    for _ in range(2):
        counts.fill_(-1), offs.fill_(-1)
        api.asap_moe_route(h, x, idx, w, counts, offs, ws)
    want = torch.bincount(idx.flatten().long(), minlength=experts)
    assert torch.equal(counts.long(), want)
    assert torch.equal(offs.long(), torch.cat([want.new_zeros(1), want.cumsum(0)]))
    # the layer's positions (from the gate's scan) and dispatch's give the same output
    out = torch.empty_like(x)
    api.asap_moe_layer(h, x, out, ws)
    xp = torch.empty((2 * n, cfg.hidden), dtype=torch.bfloat16, device=DEV)
    src, dst = torch.empty(2 * n, **i32), torch.empty((n, 2), **i32)
    y = torch.empty_like(xp)
    step = torch.empty_like(x)
    api.asap_moe_dispatch(h, x, idx, xp, src, dst, ws)
    api.asap_moe_expert_ffn(h, xp, offs, x, y, None, ws)
    api.asap_moe_combine(h, y, None, w, dst, step)
    assert api.asap_moe_status(h) == (0, 0)
    assert torch.equal(out.view(torch.int16), step.view(torch.int16))
