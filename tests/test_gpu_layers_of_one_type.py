"""Layers whose heads are all of one type: the budget of the other type, which no head of the layer has, is
exceeded at most steps, yet nothing is evicted.  Such a step takes the launches of a step that appends, and
its results are fp64 attention over all rows (bars of the parity tests: 1e-5 fp32, 2e-2 bf16 max-abs)."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("dtype,merge_last", [("f32", False), ("bf16", False), ("bf16", True)])
@pytest.mark.parametrize("contextual", [0, 1])
def test_the_budget_of_an_absent_type_changes_nothing(contextual, dtype, merge_last):
    import torch
    import paper_2504_09261_b200 as hb
    heads, dim, sides = 16, 64, (1, 2, 4, 8, 9, 30)
    total, tdt = sum(s * s for s in sides), torch.float32 if dtype == "f32" else torch.bfloat16
    mask = np.full((1, heads), contextual, dtype=np.uint8)
    caches = [hb.HackCache(1, heads, dim, 1, sides, hb.HACK_F32 if dtype == "f32" else hb.HACK_BF16, mask,
                            total if contextual else other, other if contextual else total, merge_last=merge_last)
              for other in (3, total)]
    g = torch.Generator(device="cuda").manual_seed(dim + contextual)
    ks, vs = [], []
    for k, side in enumerate(sides):
        q, kk, v = (torch.randn((1, heads, side * side, dim), generator=g, device="cuda").to(tdt) for _ in range(3))
        ks.append(kk.double())
        vs.append(v.double())
        outs, launches = [], []
        for c in caches:
            out, before = torch.full_like(q, float("nan")), c.hack_launch_count()
            c.hack_scale_step(0, k, q, kk, v, out)
            launches.append(c.hack_launch_count() - before)
            outs.append(out)
        assert launches[0] == launches[1]
        assert torch.equal(outs[0], outs[1])
        z = q.double() @ torch.cat(ks, 2).transpose(2, 3) / math.sqrt(dim)
        ref = z.softmax(-1) @ torch.cat(vs, 2)
        assert (outs[0].double() - ref).abs().max() <= (1e-5 if dtype == "f32" else 2e-2)
    for c in caches:
        assert np.array_equal(np.frombuffer(c.hack_read_head(0, 0, heads - 1, 2), dtype=np.int32), np.arange(total))
        c.close()
