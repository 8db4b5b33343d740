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
