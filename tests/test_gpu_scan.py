"""Dispatch's histogram scan over chunk ranges of one, two and several loads and
one to eight blocks of 32 experts: offsets and positions against a stable sort."""
import pytest
import torch

from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("experts", [1, 32, 33, 100, 256])
@pytest.mark.parametrize("n", [1, 33, 1025, 32769, 66000])
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
