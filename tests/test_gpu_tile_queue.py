"""CTA pairs on launches of many short tiles, where the tile queue's two slots
are reused as fast as they can be: every row bit for bit that of the single
CTAs, call after call."""
import pytest
import torch

from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("hidden,inter,n_shared", [(256, 128, 0), (2048, 128, 1)])
def test_many_short_tiles(hidden, inter, n_shared):
    cfg = inputs.small_variant(MIXTRAL, name="queue", n_experts=256, top_k=2, hidden=hidden, inter=inter,
                               n_shared=n_shared, shared_inter=128 if n_shared else 0, seed=91)
    g = torch.Generator(device=DEV).manual_seed(91)
    rows = torch.randint(0, 70, (cfg.n_experts,), generator=g, device=DEV)
    rows[7] += 600 + int(rows.sum()) % 2
    nk = int(rows.sum())
    n = nk // 2
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), n)
    offs = torch.cat([rows.new_zeros(1), rows.cumsum(0)]).to(torch.int32)
    xp = inputs.randn_bf16((nk, hidden), 1.0, 1, DEV)
    x = inputs.randn_bf16((n, hidden), 1.0, 2, DEV)
    ws = api.workspace(h, n)

    def call(mode):
        api.asap_moe_set_tiling(h, mode)
        y = torch.full((nk, hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
        ysh = torch.full((n, hidden), float("nan"), dtype=torch.bfloat16, device=DEV) if n_shared else None
        api.asap_moe_expert_ffn(h, xp, offs, x, y, ysh, ws)
        return y, ysh

    want = call(api.TILING_SINGLE)
    got = [call(api.TILING_PAIRED) for _ in range(20)]
    torch.cuda.synchronize()
    assert api.asap_moe_status(h) == (0, 0)
    for pair in got:
        for a, b in zip(pair, want):
            assert a is None or torch.equal(a.view(torch.int16), b.view(torch.int16))
    h.close()
