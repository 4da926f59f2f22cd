"""The grouped expert GEMMs on CTA pairs, on segments around the edges of
their token tiles (heights are multiples of 32, at most 256 rows, equal within
a segment): against a float64 product and, bit for bit, the single-CTA tiles."""
import pytest
import torch

from _helpers import compare_rows
from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

SEGMENTS = [
    [1, 0, 31, 32, 33, 0, 63, 64],            # heights 32 and 64, empty segments
    [65, 127, 128, 129, 255, 256, 0, 0],      # up to one full tile
    [257, 289, 511, 512, 513, 0, 7, 1],       # two and three tiles of equal height
    [0, 0, 0, 0, 0, 0, 0, 2],                 # one token
]


def _ffn64(x, wg, wu, wd):
    g = x.double() @ wg.double().t()
    h = torch.nn.functional.silu(g) * (x.double() @ wu.double().t())
    return h @ wd.double().t()


@pytest.mark.parametrize("rows", SEGMENTS, ids=lambda r: "-".join(map(str, r)))
@pytest.mark.parametrize("n_shared", [0, 1])
def test_segments_at_tile_edges(rows, n_shared):
    cfg = inputs.small_variant(MIXTRAL, name="pair", hidden=512, inter=384, n_shared=n_shared,
                               shared_inter=256 if n_shared else 0, seed=77)
    nk = sum(rows) + sum(rows) % 2
    rows = rows[:-1] + [rows[-1] + nk - sum(rows)]
    n = nk // 2
    w = inputs.make_weights(cfg, DEV)
    h = api.asap_moe_create(cfg, w, n)
    xp = inputs.randn_bf16((nk, cfg.hidden), 1.0, 1, DEV)
    x = inputs.randn_bf16((n, cfg.hidden), 1.0, 2, DEV)
    offs = torch.tensor([0] + rows, device=DEV).cumsum(0).to(torch.int32)
    outs = {}
    for mode in (api.TILING_SINGLE, api.TILING_PAIRED):
        api.asap_moe_set_tiling(h, mode)
        y = torch.full((nk, cfg.hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
        ysh = torch.full((n, cfg.hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
        api.asap_moe_expert_ffn(h, xp, offs, x, y, ysh if n_shared else None, api.workspace(h, n))
        torch.cuda.synchronize()
        outs[mode] = (y, ysh)
    assert api.asap_moe_status(h) == (0, 0)
    y, ysh = outs[api.TILING_PAIRED]
    assert torch.equal(y.view(torch.int16), outs[api.TILING_SINGLE][0].view(torch.int16))
    o = offs.tolist()
    ref = torch.cat([_ffn64(xp[o[e]:o[e + 1]], w["w_gate"][e], w["w_up"][e], w["w_down"][e])
                     for e in range(cfg.n_experts)])
    compare_rows(y.double().cpu().numpy(), ref.cpu().numpy())
    if n_shared:
        assert torch.equal(ysh.view(torch.int16), outs[api.TILING_SINGLE][1].view(torch.int16))
        compare_rows(ysh.double().cpu().numpy(),
                     _ffn64(x, w["sh_gate"], w["sh_up"], w["sh_down"]).cpu().numpy())
    h.close()
