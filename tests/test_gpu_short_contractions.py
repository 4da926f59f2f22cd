"""The bf16 expert GEMMs at contractions below 1024, where the tile kind is
chosen by K and size (one or two m-tiles per CTA, CTA pairs): the automatic
choice bit for bit the single tiles and against a float64 product, and not
slower than either kind a caller can ask for."""
import pytest
import torch

from _helpers import compare_rows
from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def _offsets(rows):
    t = torch.tensor(rows, device=DEV)
    return torch.cat([t.new_zeros(1), t.cumsum(0)]).to(torch.int32)


# gate/up K = hidden, down K = inter; large calls take the kinds named, small ones single tiles
@pytest.mark.parametrize("hidden,inter", [(256, 1024),    # two m-tiles | pairs
                                          (512, 512),     # pairs | two m-tiles
                                          (2048, 128), (2048, 384),  # pairs | two m-tiles
                                          (768, 640)])    # pairs | pairs
@pytest.mark.parametrize("rows", [[4000, 0, 1, 64, 65, 7000, 129, 9741], [6000, 2500, 2500, 2500, 2500, 2500, 2500, 2500],
                                  [300, 0, 128, 129, 1, 64, 65, 33]], ids=["ragged", "even", "small"])
def test_kinds_agree(hidden, inter, rows):
    nk, E = sum(rows), len(rows)
    n = nk // 2
    assert nk % 2 == 0
    cfg = inputs.small_variant(MIXTRAL, name="short", n_experts=E, top_k=2, hidden=hidden, inter=inter, n_shared=1,
                               shared_inter=inter, seed=41)
    w = inputs.make_weights(cfg, DEV)
    h = api.asap_moe_create(cfg, w, n)
    offs = _offsets(rows)
    xp = inputs.randn_bf16((nk, hidden), 1.0, 1, DEV)
    x = inputs.randn_bf16((n, hidden), 1.0, 2, DEV)
    outs = {}
    for mode in (api.TILING_AUTO, api.TILING_SINGLE, api.TILING_PAIRED):
        api.asap_moe_set_tiling(h, mode)
        y = torch.full((nk, hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
        ysh = torch.full((n, hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
        api.asap_moe_expert_ffn(h, xp, offs, x, y, ysh, api.workspace(h, n))
        torch.cuda.synchronize()
        outs[mode] = (y, ysh)
    assert api.asap_moe_status(h) == (0, 0)
    for mode in (api.TILING_AUTO, api.TILING_PAIRED):
        for a, b in zip(outs[mode], outs[api.TILING_SINGLE]):
            assert torch.equal(a.view(torch.int16), b.view(torch.int16))
    o = offs.tolist()
    for e in range(E):
        t = torch.arange(o[e], o[e + 1], device=DEV)
        t = t[(t - o[e] < 70) | (o[e + 1] - t <= 200)]
        if t.numel():
            g = torch.nn.functional.silu(xp[t].double() @ w["w_gate"][e].double().t())
            ref = (g * (xp[t].double() @ w["w_up"][e].double().t())) @ w["w_down"][e].double().t()
            compare_rows(outs[api.TILING_AUTO][0][t].double().cpu().numpy(), ref.cpu().numpy())
    h.close()


def _us(call):
    best = float("inf")
    for _ in range(15):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda._sleep(50_000)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


@pytest.mark.parametrize("inter", [128, 768])
def test_automatic_kind_is_not_slower(inter):
    """Many rows per expert: with single tiles at both lengths the down GEMM took
    1.24 and 1.3 times the time of the better kind."""
    hidden, E, per = 2048, 64, 2048
    nk = E * per
    cfg = inputs.small_variant(MIXTRAL, name="short_t", n_experts=E, top_k=2, hidden=hidden, inter=inter, seed=42)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), nk // 2)
    offs = _offsets([per] * E)
    hb = inputs.randn_bf16((nk, inter), 1.0, 1, DEV)
    y = torch.empty((nk, hidden), dtype=torch.bfloat16, device=DEV)
    us = {}
    for mode in (api.TILING_SINGLE, api.TILING_PAIRED, api.TILING_AUTO):
        api.asap_moe_set_tiling(h, mode)
        us[mode] = _us(lambda: api.asap_moe_expert_down(h, hb, offs, None, nk // 2, y, None))
    best = min(us[api.TILING_SINGLE], us[api.TILING_PAIRED])
    # two m-tiles are 0.82 of single tiles at K = 128; pairs 0.76 at K = 768
    assert us[api.TILING_AUTO] <= (0.93 if inter == 128 else 1.08) * best, us
    h.close()
