"""The grouped expert GEMMs on segments around the edges of their token tiles:
the bf16 CTA pairs (heights are multiples of 32, at most 256 rows, equal within
a segment) against a float64 product and, bit for bit, the single-CTA tiles;
the FP8 kernel against a float64 emulation."""
import pytest
import torch

from _helpers import compare_rows
from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import DSV3_FP8, MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"

SEGMENTS = [
    [1, 0, 31, 32, 33, 0, 63, 64],            # heights 32 and 64, empty segments
    [65, 127, 128, 129, 255, 256, 0, 0],      # up to one full tile
    [257, 289, 511, 512, 513, 0, 7, 1],       # two and three tiles of equal height
    [0, 0, 0, 0, 0, 0, 0, 2],                 # one token
    [2100, 700, 40, 33, 1, 0, 300, 260],      # bursts of many-tile segments among the others
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


def test_blocks_of_token_tiles():
    """A segment whose rows fill more than one block of the tile order (2048
    rows of 16 KB), beside a short one: every row, bit for bit."""
    cfg = inputs.small_variant(MIXTRAL, name="blocks", n_experts=2, hidden=8192, inter=256, seed=79)
    rows, n = [4500, 100], 2300
    w = inputs.make_weights(cfg, DEV)
    h = api.asap_moe_create(cfg, w, n)
    xp = inputs.randn_bf16((2 * n, cfg.hidden), 1.0, 1, DEV)
    x = inputs.randn_bf16((n, cfg.hidden), 1.0, 2, DEV)
    offs = torch.tensor([0] + rows, device=DEV).cumsum(0).to(torch.int32)
    outs = []
    for mode in (api.TILING_SINGLE, api.TILING_PAIRED):
        api.asap_moe_set_tiling(h, mode)
        y = torch.full((2 * n, cfg.hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
        api.asap_moe_expert_ffn(h, xp, offs, x, y, None, api.workspace(h, n))
        torch.cuda.synchronize()
        outs.append(y)
    assert api.asap_moe_status(h) == (0, 0)
    assert torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))
    t = torch.tensor([0, 2047, 2048, 4499, 4500, 4599], device=DEV)
    for e, sel in ((0, t[:4]), (1, t[4:])):
        compare_rows(outs[1][sel].double().cpu().numpy(),
                     _ffn64(xp[sel], w["w_gate"][e], w["w_up"][e], w["w_down"][e]).cpu().numpy())
    h.close()


def _decode(q, s):
    R, C = q.shape
    return (q.float().double().view(R // 128, 128, C // 128, 128) * s.double()[:, None, :, None]).view(R, C)


def _rows(q, s):
    return (q.float().double().view(q.shape[0], q.shape[1] // 128, 128) * s.double()[:, :, None]).view_as(q)


def _quantised(h):
    b = h.view(h.shape[0], h.shape[1] // 128, 128)
    s = b.abs().amax(dim=2, keepdim=True) / 448.0
    return ((b / s).float().to(torch.float8_e4m3fn).double() * s).view_as(h)


def _ffn_fp8(x, gate, up, down):
    a = x @ _decode(*gate).t()
    return _quantised(torch.nn.functional.silu(a) * (x @ _decode(*up).t())) @ _decode(*down).t()


@pytest.mark.parametrize("rows", SEGMENTS, ids=lambda r: "-".join(map(str, r)))
@pytest.mark.parametrize("inter", [128, 384])  # one and three K blocks of the down GEMM
def test_fp8_segments_at_tile_edges(rows, inter):
    """The FP8 GEMMs on the same segments (tiles of up to 128 rows, warps of 32)
    against a float64 emulation of the quantised product; h codes next to a
    rounding boundary may differ, hence the FP8 layer's bound over the call."""
    cfg = inputs.small_variant(DSV3_FP8, name="fp8_edges", n_experts=8, top_k=2, n_groups=1, topk_groups=1, hidden=512,
                               inter=inter, shared_inter=256, zipf_s=None, seed=78)
    nk = sum(rows) + sum(rows) % 2
    rows = rows[:-1] + [rows[-1] + nk - sum(rows)]
    n = nk // 2
    w = inputs.make_weights(cfg, DEV)
    h = api.asap_moe_create(cfg, w, n)
    g = torch.Generator(device=DEV)
    g.manual_seed(3)
    xq = torch.randn((nk, cfg.hidden), generator=g, device=DEV).mul_(100).to(torch.float8_e4m3fn)
    xs = torch.rand((nk, cfg.hidden // 128), generator=g, device=DEV) * 0.01 + 0.005
    x = inputs.randn_bf16((n, cfg.hidden), 1.0, 2, DEV)
    offs = torch.tensor([0] + rows, device=DEV).cumsum(0).to(torch.int32)
    y = torch.full((nk, cfg.hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
    ysh = torch.full((n, cfg.hidden), float("nan"), dtype=torch.bfloat16, device=DEV)
    api.asap_moe_expert_ffn(h, xq, offs, x, y, ysh, api.workspace(h, n), x_perm_scales=xs)
    torch.cuda.synchronize()
    assert api.asap_moe_status(h) == (0, 0)
    o = offs.tolist()
    kinds = ("gate", "up", "down")
    ref = torch.cat([_ffn_fp8(_rows(xq[o[e]:o[e + 1]], xs[o[e]:o[e + 1]]),
                              *((w["w_" + k][e], w["s_" + k][e]) for k in kinds)) for e in range(cfg.n_experts)])
    ref_sh = _ffn_fp8(_quantised(x.double()), *((w["sh_" + k], w["sh_s_" + k]) for k in kinds))
    for got, want in ((y.double(), ref), (ysh.double(), ref_sh)):
        # (the cast leaves a NaN code where |x| > 448: such a row is NaN on both sides, and no other is)
        nan = want.isnan().any(1)
        assert torch.equal(got.isnan().any(1), nan)
        d, r = (got - want)[~nan], want[~nan]
        assert float(d.norm() / r.norm()) <= 3e-2
        # a row's h may hold a few neighbouring codes (2^-3 apart at most); a misplaced row is off by more than 1
        assert float((d.norm(dim=1) / r.norm(dim=1)).max()) <= 0.25
    h.close()
