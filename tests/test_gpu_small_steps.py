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
