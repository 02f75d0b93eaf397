"""Small bf16 steps (one launch that appends and attends) at the edges of their tiles of 16 queries and
4 x 16 keys, against fp64 attention over the same rows.  Bar 2e-2 max-abs as in the parity tests (one
bf16 rounding of an output below 5); the appended rows are compared byte for byte."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("sides", [(1, 4, 1), (1, 1, 2, 3, 4, 5), (4, 4, 4, 4, 1, 4), (11, 4, 5, 3), (2, 30, 1, 5)])
def test_append_and_attend_over_ragged_tiles(sides, head_dim):
    import torch
    import paper_2504_09261_b200 as hb
    heads, batch, total = 3, 43, sum(s * s for s in sides)
    g = torch.Generator(device="cuda").manual_seed(total + head_dim)
    cache = hb.HackCache(1, heads, head_dim, batch, sides, hb.HACK_BF16, np.array([[1, 0, 1]], dtype=np.uint8), total, total)
    ks, vs = [], []
    for k, side in enumerate(sides):
        q, kk, v = (torch.randn((batch, heads, side * side, head_dim), generator=g, device="cuda").bfloat16() for _ in range(3))
        ks.append(kk)
        vs.append(v)
        out = torch.full_like(q, float("nan"))
        cache.hack_scale_step(0, k, q, kk, v, out)
        z = q.double() @ torch.cat(ks, 2).double().transpose(2, 3) / math.sqrt(head_dim)
        ref = z.softmax(-1) @ torch.cat(vs, 2).double()
        assert (out.double() - ref).abs().max() <= 2e-2
    for b, h in ((0, 0), (batch - 1, heads - 1)):
        for which, rows in ((0, ks), (1, vs)):
            want = torch.cat(rows, 2)[b, h].contiguous().view(torch.uint8).cpu().numpy().tobytes()
            assert cache.hack_read_head(0, b, h, which) == want
        assert np.array_equal(np.frombuffer(cache.hack_read_head(0, b, h, 2), dtype=np.int32), np.arange(total))
    cache.close()


@pytest.mark.parametrize("base,heads,batch,sides,b_c,b_s,policy", [
    (1, 5, 1, (1, 2, 3, 5, 7, 9), 47, 128, 0),              # up to 128 ranked candidates, every CTA one row tile
    (1, 16, 1, (1, 2, 6, 10, 13), 87, 255, 1),              # 256 = two key tiles per warp; the current scale competes
    (1, 8, 1, (1, 2, 7, 13, 15), 60, 287, 0),               # 512 = four, clusters of eight
    (1, 4, 1, (1, 2, 9, 15, 19), 50, 407, 1),               # 768 = six
    (1, 30, 8, (1, 2, 4, 6, 7), 39, 101, 0),                # 240 heads, two CTAs per SM
    (1, 7, 3, (5, 5, 1, 1, 4), 20, 33, 1),                  # steps of a single token that evict
    (3, 16, 1, (1, 3, 5, 8, 9), 33, 97, 0),                 # head_dim 128
    (3, 9, 2, (1, 2, 8, 12), 1, 150, 1),                    # a contextual head keeps one row
])
def test_whole_step_in_one_launch(base, heads, batch, sides, b_c, b_s, policy):
    from dataclasses import replace
    from parity_util import run_parity
    from workloads import get_config
    cfg = replace(get_config(base, n_layers=1), name=f"small-{heads}x{batch}", n_heads=heads, batch=batch, sides=sides,
                  budget_c=b_c, budget_s=b_s)
    rep = run_parity(cfg, [0], fused=True, policy=policy)
    assert rep.ok(), rep.problems[:5]
    assert rep.compressed_heads > 0
    assert set(rep.evicting_launches) == {1}, rep.evicting_launches


@pytest.mark.parametrize("head_dim", [64, 128])
def test_equal_scores_in_one_launch(head_dim):
    """All keys zero: every entry lies in the located bin and the lowest candidate indices survive; the
    outputs are the mean of the survivors' values (bar as above).  Every step is one launch."""
    import torch
    import paper_2504_09261_b200 as hb
    sides, b_c, b_s, heads = (2, 3, 5, 9), 21, 100, 6
    mask = np.array([[h % 2 for h in range(heads)]], dtype=np.uint8)
    cache = hb.HackCache(1, heads, head_dim, 1, sides, hb.HACK_BF16, mask, b_c, b_s)
    kept, total = [[], []], 0
    for k, side in enumerate(sides):
        n = side * side
        z = torch.zeros((1, heads, n, head_dim), dtype=torch.bfloat16, device="cuda")
        v = (torch.arange(total, total + n, device="cuda") / 128).bfloat16()[None, None, :, None].expand_as(z).contiguous()
        out = torch.empty_like(z)
        before = cache.hack_launch_count()
        cache.hack_scale_step(0, k, torch.randn_like(z), z, v, out)
        assert cache.hack_launch_count() == before + 1
        new = list(range(total, total + n))
        total += n
        for t, budget in ((0, b_s), (1, b_c)):
            cand = kept[t] + new
            if len(cand) > budget and t == 0:               # the leading two scales and the new one are protected
                cand = cand[:max(budget, 13 + n) - n] + new
            kept[t] = cand if t == 0 else cand[:budget]
        for h in range(heads):
            t = int(mask[0, h])
            assert np.array_equal(np.frombuffer(cache.hack_read_head(0, 0, h, 2), dtype=np.int32), kept[t])
            mean = (torch.tensor(kept[t], device="cuda") / 128).bfloat16().double().mean()
            assert (out[0, h].double() - mean).abs().max() <= 2e-2
    cache.close()


@pytest.mark.parametrize("head_dim,heads,batch,sides,b_c,b_s,policy", [
    (64, 5, 1, (1, 2, 3, 5, 7), 29, 63, 0),                 # up to two groups of 32 keys per warp, ragged last tile
    (64, 16, 1, (1, 2, 6, 10, 10), 87, 156, 1),             # 187 and 256 candidates: four groups
    (64, 9, 2, (1, 2, 7, 11, 15), 95, 95, 1),               # 320 candidates: five, the largest served
    (64, 30, 5, (1, 2, 4, 6), 39, 41, 0),                   # 150 heads, two CTAs per SM
    (64, 7, 3, (5, 5, 1, 1, 4), 20, 33, 1),                 # steps of a single token that evict
    (128, 6, 2, (1, 3, 5, 8, 9), 1, 97, 0),                 # head_dim 128; contextual heads keep one row
])
def test_whole_fp32_step_in_one_launch(head_dim, heads, batch, sides, b_c, b_s, policy):
    from dataclasses import replace
    from parity_util import run_parity
    from workloads import get_config
    cfg = replace(get_config(0), name=f"small-f32-{heads}x{batch}", n_heads=heads, batch=batch, head_dim=head_dim, sides=sides,
                  budget_c=b_c, budget_s=b_s)
    rep = run_parity(cfg, [0], fused=True, policy=policy)
    assert rep.ok(), rep.problems[:5]
    assert rep.compressed_heads > 0
    assert set(rep.evicting_launches) == {1}, rep.evicting_launches
