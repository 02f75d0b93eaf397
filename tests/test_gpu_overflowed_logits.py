"""Keys whose logits are -inf (a product that overflowed) weigh nothing, wherever they lie: as the only key
a warp or a tile has, as the whole new scale, in steps that append and in steps that evict in one launch.

Every query has 1 and every such key -inf in dimension 0.  The reference is fp64 attention over the rows
that the cache holds afterwards; bars as in the parity tests (1e-5 fp32, 2e-2 bf16 max-abs)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


# (sides, heads, budgets, positions of the overflowing keys at each scale)
SHAPES = [
    ((4, 1), 2, (99, 99), {1: [0]}),                                    # 17 keys: the last one alone in a warp's share
    ((4, 5, 3), 3, (99, 99), {1: range(0, 25, 2), 2: range(9)}),        # 50 keys, the new scale overflows as a whole
    ((5, 2, 2), 2, (99, 99), {1: range(4), 2: range(4)}),               # 33 keys: one past a tile of 32
    ((6, 12), 32, (999, 999), {1: range(128)}),                         # the first tile of 128 rows of the new scale
    ((1, 2, 3, 5, 7), 5, (29, 63), {4: range(49)}),                     # evicting: protected rows that weigh nothing
    ((1, 2, 6, 10), 16, (40, 120), {3: range(3, 100)}),
]


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("sides,heads,budgets,bad", SHAPES)
def test_overflowed_logits_weigh_nothing(sides, heads, budgets, bad, head_dim, dtype):
    import torch
    import paper_2504_09261_b200 as hb
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    mask = (np.arange(heads) % 2).astype(np.uint8)[None]
    caches = [hb.HackCache(1, heads, head_dim, 1, sides, hb.HACK_F32 if dtype == "f32" else hb.HACK_BF16, mask, *budgets)
              for _ in range(2)]
    g = torch.Generator(device="cuda").manual_seed(sum(sides) + head_dim)
    ks = torch.empty((heads, 0, head_dim), device="cuda", dtype=torch.float64)
    vs = ks.clone()
    for k, side in enumerate(sides):
        q, kk, v = (torch.randn((1, heads, side * side, head_dim), generator=g, device="cuda") for _ in range(3))
        q[..., 0] = 1.0
        kk[:, :, list(bad.get(k, [])), 0] = -math.inf
        q, kk, v = q.to(tdt), kk.to(tdt), v.to(tdt)
        ks, vs = torch.cat([ks, kk[0].double()], 1), torch.cat([vs, v[0].double()], 1)
        fused, staged = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
        info = caches[0].hack_step_info(0, k)
        caches[0].hack_scale_step(0, k, q, kk, v, fused)
        outs = [(0, fused)]
        if not (info.triggered_c or info.triggered_s):                  # the stage calls, as far as nothing is evicted
            idx = torch.zeros((heads, caches[1].kept_stride), dtype=torch.int32, device="cuda")
            scores = torch.zeros((heads, caches[1].cand_stride), device="cuda")
            caches[1].hack_select(0, k, scores, idx)
            caches[1].hack_compact(0, k, idx, kk, v)
            caches[1].hack_attend(0, k, q, staged)
            outs.append((1, staged))
        for which, out in outs:
            for h in range(heads):
                pos = torch.from_numpy(np.frombuffer(caches[which].hack_read_head(0, 0, h, 2), dtype=np.int32).astype(np.int64)).cuda()
                z = q[0, h].double() @ ks[h, pos].T / math.sqrt(head_dim)
                ref = z.softmax(-1) @ vs[h, pos]
                assert bool(torch.isfinite(ref).all())
                err = (out[0, h].double() - ref).abs().max()
                assert bool(err <= (1e-5 if dtype == "f32" else 2e-2)), (which, k, h, float(err))
    for c in caches:
        c.close()
