"""dispatch and combine of rows of every width class (several tokens per CTA up
to rows of 512 vectors), with token counts that leave a CTA, a chunk or a warp
partly filled, against a stable sort and a float64 sum; the mailbox's forms
against the layer call."""
import pytest
import torch

from _helpers import compare_rows
from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import DSV3_FP8, MIXTRAL

pytestmark = pytest.mark.gpu
DEV = "cuda:0"
I32 = dict(dtype=torch.int32, device=DEV)
F8 = dict(n_groups=1, topk_groups=1, shared_inter=128, zipf_s=None)


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


@pytest.mark.parametrize("hidden", [256, 512, 768, 1536, 1792, 2048, 4096, 4352])
@pytest.mark.parametrize("n,k", [(1, 8), (31, 3), (33, 8), (457, 1), (1001, 8)])
def test_dispatch_and_combine(hidden, n, k):
    cfg = inputs.small_variant(MIXTRAL, name="narrow", hidden=hidden, inter=128, n_experts=24, top_k=k, seed=31)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), n)
    g = torch.Generator(device=DEV).manual_seed(n)
    # every expert of a token once, the low ones often
    score = torch.rand((n, 24), generator=g, device=DEV) - torch.arange(24, device=DEV) / 24
    idx = score.topk(k, dim=1).indices.to(torch.int32).contiguous()
    x = inputs.randn_bf16((n, hidden), 1.0, 1, DEV)
    xp = torch.empty((n * k, hidden), dtype=torch.bfloat16, device=DEV)
    src, dst = torch.full((n * k,), -1, **I32), torch.full((n, k), -1, **I32)
    api.asap_moe_dispatch(h, x, idx, xp, src, dst, api.workspace(h, n))
    order = torch.sort(idx.flatten().long(), stable=True).indices
    assert torch.equal(dst.flatten().long()[order], torch.arange(n * k, device=DEV))
    assert torch.equal(src.long(), order // k)
    assert torch.equal(xp.view(torch.int16), x[order // k].view(torch.int16))
    w = torch.rand((n, k), generator=g, device=DEV)
    out = torch.full_like(x, float("nan"))
    api.asap_moe_combine(h, xp, None, w, dst, out)
    assert api.asap_moe_status(h) == (0, 0)
    ref = (xp.double()[dst.long()] * w.double()[:, :, None]).sum(1)
    compare_rows(out.double().cpu().numpy(), ref.cpu().numpy())
    h.close()


@pytest.mark.parametrize("hidden", [256, 768, 2048])
def test_dispatch_fp8(hidden):
    n, k = 301, 5
    cfg = inputs.small_variant(DSV3_FP8, name="narrow8", hidden=hidden, inter=128, n_experts=24, top_k=k, seed=32, **F8)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), n)
    g = torch.Generator(device=DEV).manual_seed(2)
    idx = torch.rand((n, 24), generator=g, device=DEV).topk(k, dim=1).indices.to(torch.int32).contiguous()
    x = inputs.randn_bf16((n, hidden), 1.0, 1, DEV)
    xp = torch.empty((n * k, hidden), dtype=torch.float8_e4m3fn, device=DEV)
    xs = torch.empty((n * k, hidden // 128), device=DEV)
    src, dst = torch.full((n * k,), -1, **I32), torch.full((n, k), -1, **I32)
    api.asap_moe_dispatch(h, x, idx, xp, src, dst, api.workspace(h, n), x_perm_scales=xs)
    assert api.asap_moe_status(h) == (0, 0)
    order = torch.sort(idx.flatten().long(), stable=True).indices
    assert torch.equal(src.long(), order // k)
    b = x[order // k].double().view(n * k, hidden // 128, 128)
    amax = b.abs().amax(2)
    torch.testing.assert_close(xs.double(), amax / 448.0, rtol=2.0 ** -22, atol=0)
    # half an e4m3 step of the block's largest value (2^-4 of it) bounds every value's error
    err = (xp.double().view_as(b) * xs.double()[:, :, None] - b).abs()
    assert bool((err <= amax[:, :, None] * 2.0 ** -4 * 1.001).all())
    h.close()


@pytest.mark.parametrize("base,hidden", [(MIXTRAL, 256), (MIXTRAL, 1024), (DSV3_FP8, 512)],
                         ids=["bf16_256", "bf16_1024", "fp8_512"])
def test_mailbox_posts_of_partial_groups(base, hidden):
    extra = F8 if base is DSV3_FP8 else {}
    cfg = inputs.small_variant(base, name="narrow_mb", hidden=hidden, inter=128, n_experts=16, top_k=4, seed=33, **extra)
    sizes = [3, 129, 31, 300]
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), 300)
    box = api.asap_moe_mailbox_create(h, len(sizes), 300)
    xs = [inputs.make_tokens(cfg, n, i, DEV) for i, n in enumerate(sizes)]
    outs = [torch.full_like(x, float("nan")) for x in xs]
    epochs = [api.asap_moe_mailbox_post(box, i, x, o) for i, (x, o) in enumerate(zip(xs, outs))]
    api.asap_moe_mailbox_serve_many(box, list(range(len(sizes))), epochs)
    for i in range(len(sizes)):
        api.asap_moe_mailbox_wait(box, i)
    torch.cuda.synchronize()
    assert api.asap_moe_status(h) == (0, 0)
    for x, o in zip(xs, outs):
        ref = torch.empty_like(x)
        api.asap_moe_layer(h, x, ref, api.workspace(h, x.shape[0]))
        assert torch.equal(o.view(torch.int16), ref.view(torch.int16))
    box.close()
    h.close()


def _us(call):
    best = float("inf")
    for _ in range(20):
        a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
        torch.cuda._sleep(50_000)
        a.record()
        call()
        b.record()
        torch.cuda.synchronize()
        best = min(best, a.elapsed_time(b) * 1e3)
    return best


def test_many_narrow_rows_are_bound_by_their_bytes():
    """65536 tokens of 256 channels: a warp per token takes about twice the time
    of a copy of the same bytes, a CTA per token four (dispatch) to six times
    (combine); the bound lies between."""
    n, k, hidden = 65536, 8, 256
    cfg = inputs.small_variant(MIXTRAL, name="narrow_t", hidden=hidden, inter=128, n_experts=64, top_k=k, seed=34)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), n)
    g = torch.Generator(device=DEV).manual_seed(1)
    idx = torch.rand((n, 64), generator=g, device=DEV).topk(k, dim=1).indices.to(torch.int32).contiguous()
    x = inputs.randn_bf16((n, hidden), 1.0, 1, DEV)
    xp = torch.empty((n * k, hidden), dtype=torch.bfloat16, device=DEV)
    src, dst = torch.empty(n * k, **I32), torch.empty((n, k), **I32)
    ws, w, out = api.workspace(h, n), torch.rand((n, k), device=DEV), torch.empty_like(x)
    api.asap_moe_dispatch(h, x, idx, xp, src, dst, ws)
    both = torch.empty((n * (k + 1) // 2, hidden), dtype=torch.bfloat16, device=DEV)  # read once, written once
    other = torch.empty_like(both)
    copy = _us(lambda: other.copy_(both))
    dispatch = _us(lambda: api.asap_moe_dispatch(h, x, idx, xp, src, dst, ws))
    combine = _us(lambda: api.asap_moe_combine(h, xp, None, w, dst, out))
    assert dispatch <= 3 * copy and combine <= 3 * copy, (copy, dispatch, combine)
    h.close()
