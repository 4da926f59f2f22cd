"""Calls enqueued back to back on one stream and one workspace, with other
inputs and other token counts each time and no synchronisation between them: a
kernel that read what the call before left in the workspace (histogram, chunk
bases, positions, rows) would give the wrong output.  Each output must equal,
bit for bit, that of the same call alone on a workspace of its own."""
import pytest
import torch

from paper_2606_22541_gb300 import api, inputs
from paper_2606_22541_gb300.configs import DSV3, DSV3_FP8, MIXTRAL, TINY

pytestmark = pytest.mark.gpu
DEV = "cuda"
# one-launch route or gate with scan, CTA pairs or single CTAs, FP8
DS = inputs.small_variant(DSV3, name="dep_ds", hidden=1024, inter=256, shared_inter=256, microbatches=[700])
MX = inputs.small_variant(MIXTRAL, name="dep_mx", hidden=1024, inter=1024, microbatches=[700])
F8 = inputs.small_variant(DSV3_FP8, name="dep_f8", hidden=512, inter=256, shared_inter=256, microbatches=[700])
SIZES = [257, 33, 700, 1, 512, 96, 700, 65]
ROUNDS = 6


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__
    __graft_entry__.build()


def same_bits(a, b):
    return torch.equal(a.view(torch.int16), b.view(torch.int16))


@pytest.mark.parametrize("cfg", [TINY, DS, MX, F8], ids=lambda c: c.name)
def test_layers_with_other_inputs_on_one_workspace(cfg):
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), max(SIZES))
    xs = [inputs.make_tokens(cfg, n, i, DEV) for i, n in enumerate(SIZES)]
    want = []
    for x in xs:
        out = torch.empty_like(x)
        api.asap_moe_layer(h, x, out, api.workspace(h, x.shape[0]))
        torch.cuda.synchronize()
        want.append(out)
    ws = api.workspace(h, max(SIZES))
    got = [[torch.full_like(x, 7.0) for x in xs] for _ in range(ROUNDS)]
    torch.cuda.synchronize()
    for outs in got:
        for x, out in zip(xs, outs):
            api.asap_moe_layer(h, x, out, ws)
    torch.cuda.synchronize()
    assert api.asap_moe_status(h) == (0, 0)
    for outs in got:
        for n, out, ref in zip(SIZES, outs, want):
            assert same_bits(out, ref), n


@pytest.mark.parametrize("sizes", [[257, 33, 256, 1], [8193, 1025, 8192, 31]], ids=str)
def test_steps_with_other_inputs_on_one_workspace(sizes):
    """route and dispatch across the sizes at which their launches change."""
    cfg = inputs.small_variant(MIXTRAL, name="dep_steps", hidden=256, inter=256, n_experts=64, top_k=2, seed=9)
    h = api.asap_moe_create(cfg, inputs.make_weights(cfg, DEV), max(sizes))
    i32 = dict(dtype=torch.int32, device=DEV)

    def buffers(n):
        return dict(idx=torch.full((n, 2), -1, **i32), w=torch.empty((n, 2), device=DEV),
                    counts=torch.full((64,), -1, **i32), offs=torch.full((65,), -1, **i32),
                    xp=torch.empty((2 * n, 256), dtype=torch.bfloat16, device=DEV), src=torch.full((2 * n,), -1, **i32),
                    dst=torch.full((n, 2), -1, **i32))

    def call(x, b, ws):
        api.asap_moe_route(h, x, b["idx"], b["w"], b["counts"], b["offs"], ws)
        api.asap_moe_dispatch(h, x, b["idx"], b["xp"], b["src"], b["dst"], ws)

    xs = [inputs.make_tokens(cfg, n, i, DEV) for i, n in enumerate(sizes)]
    ws = api.workspace(h, max(sizes))
    got = [[buffers(n) for n in sizes] for _ in range(ROUNDS)]
    torch.cuda.synchronize()
    for bs in got:
        for x, b in zip(xs, bs):
            call(x, b, ws)
    torch.cuda.synchronize()
    assert api.asap_moe_status(h) == (0, 0)
    for i, (n, x) in enumerate(zip(sizes, xs)):
        ref = buffers(n)
        call(x, ref, api.workspace(h, n))
        torch.cuda.synchronize()
        order = torch.sort(ref["idx"].flatten().long(), stable=True).indices
        assert torch.equal(ref["src"].long(), order // 2) and same_bits(ref["xp"], x[order // 2])
        for bs in got:
            assert all(torch.equal(bs[i][key], ref[key]) for key in ref), n
