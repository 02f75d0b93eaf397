"""More (batch, head) pairs than a grid's second dimension holds: steps that append, from a first scale that
the tensor-core attention serves.  A sample of heads against fp64 attention, bar 2e-2 max-abs as in the
parity tests of bf16 outputs."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


def test_appending_steps_of_more_than_65535_heads():
    import torch
    import paper_2504_09261_b200 as hb
    heads, batch, sides, dim = 7, 9400, (6, 6), 64
    mask = (np.arange(heads) % 2).astype(np.uint8)[None]
    cache = hb.HackCache(1, heads, dim, batch, sides, hb.HACK_BF16, mask, 72, 72)
    g = torch.Generator(device="cuda").manual_seed(65536)
    ks, vs = [], []
    for k, side in enumerate(sides):
        q, kk, v = (torch.randn((batch, heads, side * side, dim), generator=g, device="cuda").bfloat16() for _ in range(3))
        ks.append(kk)
        vs.append(v)
        out = torch.full_like(q, float("nan"))
        cache.hack_scale_step(0, k, q, kk, v, out)
        assert bool(torch.isfinite(out).all())
        for b, h in ((0, 0), (1, 6), (4700, 3), (9362, 1), (9399, 6)):
            kc, vc = (torch.cat([t[b, h].double() for t in part]) for part in (ks, vs))
            ref = (q[b, h].double() @ kc.T / math.sqrt(dim)).softmax(-1) @ vc
            assert (out[b, h].double() - ref).abs().max() <= 2e-2
    cache.close()
