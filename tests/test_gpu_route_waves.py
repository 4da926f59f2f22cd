"""Routing with the CUDA-core router in more than one wave of CTAs: the gate and
scan behind it must not slow it down.  A call takes 1.29 (100 experts) and 1.17
(128) times the time of its logits; with the gate's CTAs resident beside the
router's last wave it took 1.57 and 1.52.  The bounds lie half-way."""
import pytest
import torch

from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda"


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _us(call):
    best = float("inf")
    for _ in range(25):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda._sleep(50_000)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


@pytest.mark.parametrize("experts,bound", [(100, 1.43), (128, 1.34)])
def test_route_of_two_waves(experts, bound):
    n, i32 = 4096, dict(dtype=torch.int32, device=DEV)
    cfg = inputs.small_variant(MIXTRAL, name="waves", hidden=256, inter=128, n_experts=experts, top_k=4, seed=4)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), n)
    ws, x = api.workspace(h, n), inputs.make_tokens(cfg, n, 0, DEV)
    idx, w = torch.empty((n, 4), **i32), torch.empty((n, 4), device=DEV)
    counts, offs = torch.empty(experts, **i32), torch.empty(experts + 1, **i32)
    logits = torch.empty((n, experts), device=DEV)
    router = _us(lambda: api.asap_moe_router_logits(h, x, logits, ws))
    route = _us(lambda: api.asap_moe_route(h, x, idx, w, counts, offs, ws))
    assert route <= bound * router, (router, route)
    h.close()
