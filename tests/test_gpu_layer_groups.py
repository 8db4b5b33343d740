"""cc_compress_layers where the layers fill one launch exactly, spill into another, or are many
sequences each: indices are those of separate calls (up to ties that f32 rounding decides), and the
rows gathered are exactly those that the indices name."""
import pytest
import torch

from paper_2604_10235_b200 import binding as cc
from paper_2604_10235_b200 import inputs as gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("layers,w,lens", [(32, 16, (300,)), (33, 16, (300,)), (65, 32, (129,)),
                                           (7, 16, (40, 513, 200) * 7)])
def test_groups_of_layers_equal_separate_calls(layers, w, lens):
    from gpu_util import bf16_dev, ctx, desc_for
    wl = gen.Workload("groups", 41, 1, 8, 2, 128, w, gen.POOL_MAX, 7, 0, seq_lens=lens, budget_frac=0.2)
    xs = [gen.make_layer(wl, layer=l) for l in range(3)]
    d = desc_for(wl, cc.CC_MODE_BF16)
    ws, prior = ctx().workspace(d), torch.from_numpy(xs[0].prior).cuda()
    q, k, v = ([bf16_dev(getattr(xs[l % 3], a)) for l in range(layers)] for a in ("q_win", "k", "v"))
    b_tot, n_seq = sum(wl.budgets), len(wl.lens)

    def outputs(n):
        ko = [torch.zeros((b_tot, 2, 128), dtype=torch.bfloat16, device="cuda") for _ in range(n)]
        return (ko, [torch.zeros_like(t) for t in ko],
                [torch.full((2, b_tot), -9, dtype=torch.int32, device="cuda") for _ in range(n)],
                [torch.full((n_seq, 2), -9, dtype=torch.int32, device="cuda") for _ in range(n)])

    one, all_ = outputs(3), outputs(layers)
    for l in range(3):
        cc.cc_compress_layer(ctx(), d, q[l], k[l], v[l], prior, *(t[l] for t in one), None, None, ws)
    cc.cc_compress_layers(ctx(), d, q, k, v, prior, *all_, None, None, ws)
    assert ctx().poll() == 0
    starts = torch.tensor([sum(wl.lens[:s]) for s in range(n_seq)], device="cuda")
    base = torch.repeat_interleave(starts, torch.tensor(wl.budgets, device="cuda"))   # first token of a slot's sequence
    for l in range(layers):
        ko, vo, idx, count = (t[l] for t in all_)
        assert torch.equal(count, one[3][l % 3])
        assert (idx != one[2][l % 3]).float().mean() <= 0.01
        for h in range(2):
            rows = base + idx[h]
            assert torch.equal(ko[:, h].view(torch.int16), k[l][rows, h].view(torch.int16))
            assert torch.equal(vo[:, h].view(torch.int16), v[l][rows, h].view(torch.int16))


@pytest.mark.parametrize("shared", ["idx", "idx_and_count", "all_outputs", "previous_k", "previous_v", "free_list",
                                    "interleaved", "interleaved_in_place"])
def test_layers_that_share_buffers(shared):
    """What layers compute when they run one after the other, bit for bit where the sharing makes them run
    so, whoever shares what: scratch outputs, caches compacted into the space of the layer before, one page
    list; caches interleaved row by row share nothing."""
    from gpu_util import bf16_dev, ctx, desc_for
    paged = shared in ("free_list", "interleaved_in_place")
    wl = gen.Workload("share", 43, 1, 8, 2, 128, 32, gen.POOL_MAX, 7, 0, seq_lens=(700, 300), budget_frac=0.4,
                      page_size=16 if paged else 0)
    layers, hkv, b_tot = 5, 2, sum(wl.budgets)
    xs = [gen.make_layer(wl, layer=l) for l in range(layers)]
    if paged:
        for x in xs[1:]:
            gen.repage(x, xs[0])
    rows = xs[0].k.shape[0]
    stride = max(-(-b // 16) for b in wl.budgets) if paged else 0
    woven = shared.startswith("interleaved")
    pt = torch.from_numpy(xs[0].page_table).cuda() if paged else None
    d = desc_for(wl, cc.CC_MODE_BF16, page_table=pt, out_pt_stride=stride, pool_pages=xs[0].pool_pages)
    if woven:                                    # [token][layer][head][channel]
        d.c.kv_stride_tok = d.c.out_stride_tok = layers * hkv * 128
    prior = torch.from_numpy(xs[0].prior).cuda()
    q = [bf16_dev(x.q_win) for x in xs]

    def cache(attr):
        made = [bf16_dev(getattr(x, attr)) for x in xs]
        return list(torch.stack(made, 1).unbind(1)) if woven else made

    def empty_cache():
        if woven:
            return list(torch.zeros((b_tot, layers, hkv, 128), dtype=torch.bfloat16, device="cuda").unbind(1))
        return [torch.zeros((b_tot, hkv, 128), dtype=torch.bfloat16, device="cuda") for _ in xs]

    def buffers():
        k, v = cache("k"), cache("v")
        ko, vo = (k, v) if paged else (empty_cache(), empty_cache())
        idx = [torch.full((hkv, b_tot), -9, dtype=torch.int32, device="cuda") for _ in xs]
        count = [torch.full((2, hkv), -9, dtype=torch.int32, device="cuda") for _ in xs]
        free = opt = None
        if paged:
            free = [torch.from_numpy(xs[0].free_pages).cuda()] * layers
            opt = [torch.full((2, stride), -9, dtype=torch.int32, device="cuda")] * layers
        if shared.startswith("idx") or shared == "all_outputs":
            idx = idx[:1] * layers
        if shared in ("idx_and_count", "all_outputs"):
            count = count[:1] * layers
        if shared == "all_outputs":
            ko, vo = ko[:1] * layers, vo[:1] * layers
        if shared == "previous_k":               # the last layer's into a buffer of its own
            ko = [ko[0]] + [t[:b_tot] for t in k[:-1]]
        if shared == "previous_v":
            vo = [vo[0]] + [t[100:100 + b_tot] for t in v[:-1]]
        return k, v, ko, vo, idx, count, free, opt

    one, all_ = buffers(), buffers()
    ws = ctx().workspace(d)
    for l in range(layers):
        cc.cc_compress_layer(ctx(), d, q[l], *(t[l] for t in one[:2]), prior, *(t[l] if t else None for t in one[2:]), ws)
    assert ctx().poll() == 0
    cc.cc_compress_layers(ctx(), d, q, *all_[:2], prior, *all_[2:], ws)
    assert ctx().poll() == 0
    together = paged or woven                    # several layers to a launch: ties that f32 rounding decides may swap
    for a, b in zip(one, all_):
        for s, t in zip(a or [], b or []):
            if s.dtype == torch.bfloat16:
                s, t = s.view(torch.int16), t.view(torch.int16)
            assert torch.equal(s, t) or (together and (s != t).float().mean() <= 0.01)


@pytest.mark.parametrize("layers,room", [(7, 1), (7, 2), (7, 3), (7, 7), (33, 33), (40, 33), (1, 1)])
def test_workspace_of_some_layers(layers, room):
    """One layer's workspace is what its own call needs; cc_compress_layers keeps inside what it is given, be that
    one layer's, some layers' or all layers', and refuses less than one layer's."""
    from gpu_util import bf16_dev, ctx, desc_for
    wl = gen.Workload("room", 44, 1, 8, 2, 128, 32, gen.POOL_MAX, 7, 300, n=1500)
    xs = [gen.make_layer(wl, layer=l) for l in range(3)]
    d = desc_for(wl, cc.CC_MODE_BF16)
    n_bytes = ctx().workspace_bytes(d, room)
    one_layer = ctx().workspace_bytes(d, 1)
    stats = 256 * 8 * 150                        # (maximum, sum) of 128 rows per CTA and (sequence, head)
    assert one_layer <= 2 * 4 * 2 * 1500 + stats + 2 * 1500 + 4 * 256 and one_layer <= n_bytes <= ctx().workspace_bytes(d)
    assert ctx().lib.cc_workspace_bytes(ctx().handle, d.c) == one_layer
    full = torch.full((n_bytes + 4096,), 0x5A, dtype=torch.uint8, device="cuda")
    prior = torch.from_numpy(xs[0].prior).cuda()
    q, k, v = ([bf16_dev(getattr(xs[l % 3], a)) for l in range(layers)] for a in ("q_win", "k", "v"))

    def outputs(n):
        ko = torch.zeros((n, 300, 2, 128), dtype=torch.bfloat16, device="cuda")
        return (list(ko), list(torch.zeros_like(ko)),
                list(torch.full((n, 2, 300), -9, dtype=torch.int32, device="cuda")),
                list(torch.full((n, 1, 2), -9, dtype=torch.int32, device="cuda")))

    one, all_ = outputs(3), outputs(layers)
    for l in range(3):
        cc.cc_compress_layer(ctx(), d, q[l % layers], k[l % layers], v[l % layers], prior, *(t[l] for t in one))
    cc.cc_compress_layers(ctx(), d, q, k, v, prior, *all_, ws=full[:n_bytes])
    assert ctx().poll() == 0
    assert bool((full[n_bytes:] == 0x5A).all())
    for l in range(layers):
        same = [torch.equal(s[l].view(torch.int16), t[l % 3].view(torch.int16)) for s, t in zip(all_, one)]
        assert all(same) or (room > 1 and (all_[2][l] != one[2][l % 3]).float().mean() <= 0.01)
    with pytest.raises(cc.CodecompError) as e:
        cc.cc_compress_layers(ctx(), d, q, k, v, prior, *all_, ws=full[:one_layer - 256])
    assert e.value.status == cc.CC_ERR_WORKSPACE
