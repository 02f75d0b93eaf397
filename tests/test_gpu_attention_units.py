"""The tensor-core attention at the edges of its work split: last blocks of a segment of every number of 32-key
groups (the caller's rows and the cache's), more units than CTAs run at once (a CTA takes over units that were not
launched), and heads whose keys are one block (several rounds of query tiles per unit).  Heads are compared with
64-bit attention over the rows the cache reports; bar 2e-2 max-abs as in the parity tests of bf16 outputs."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


def decode(dim, heads, batch, sides, b_c, b_s, sample):
    import torch
    import paper_2504_09261_b200 as hb
    mask = (np.arange(heads) % 2).astype(np.uint8)[None]
    cache = hb.HackCache(1, heads, dim, batch, sides, hb.HACK_BF16, mask, b_c, b_s)
    g = torch.Generator(device="cuda").manual_seed(dim + heads)
    ks, vs = [], []
    for k, side in enumerate(sides):
        q, kk, v = (torch.randn((batch, heads, side * side, dim), generator=g, device="cuda").bfloat16() for _ in range(3))
        ks.append(kk)
        vs.append(v)
        out = torch.full_like(q, float("nan"))
        cache.hack_scale_step(0, k, q, kk, v, out)
        assert bool(torch.isfinite(out).all())
        for b, h in sample:
            pos = torch.from_numpy(np.frombuffer(cache.hack_read_head(0, b, h, 2), dtype=np.int32).copy()).long().cuda()
            kc, vc = (torch.cat([t[b, h] for t in part])[pos].double() for part in (ks, vs))
            ref = (q[b, h].double() @ kc.T / math.sqrt(dim)).softmax(-1) @ vc
            err = (out[b, h].double() - ref).abs().max().item()
            assert err <= 2e-2, (side, b, h, len(pos), err)
    cache.hack_poll_status()
    cache.close()


# tokens modulo 128: 17 -> 16, 21 -> 57, 15 -> 97, 31 -> 65, 24 -> 64, 23 -> 17, 22 -> 100, 20 -> 16, 30 -> 4, 16 -> 0
@pytest.mark.parametrize("dim,heads,batch,sides", [
    (64, 3, 1, (15, 17, 31)), (64, 2, 2, (24, 23, 21)), (64, 5, 60, (15, 16, 17)),
    (128, 3, 1, (15, 17, 31)), (128, 2, 2, (24, 23, 21)), (128, 9, 12, (22, 20, 30)), (128, 2, 100, (16, 31)),
])
def test_last_blocks_of_both_segments(dim, heads, batch, sides):
    total = sum(s * s for s in sides)
    decode(dim, heads, batch, sides, total, total, [(0, 0), (batch - 1, heads - 1)])


@pytest.mark.parametrize("dim,heads,batch,sides,b_c,b_s", [
    (64, 16, 16, (2, 8, 20, 32), 33, 1045),      # contextual heads of one short block, 6 rounds of one tile
    (128, 12, 10, (2, 9, 33, 40), 100, 1700),    # the same on two tiles, an odd number of rounds
    (64, 30, 12, (3, 9, 21, 24), 128, 700),      # a whole block
    (128, 30, 8, (2, 7, 18, 29), 230, 900),      # more units than SMs, behind a compression
])
def test_rounds_and_units_that_change_hands(dim, heads, batch, sides, b_c, b_s):
    decode(dim, heads, batch, sides, b_c, b_s, [(0, 0), (0, 1), (batch // 2, heads - 1), (batch - 1, heads - 2)])


@pytest.mark.parametrize("dim,sides", [(64, (2, 9, 21)), (64, (3, 20, 40)), (128, (2, 9, 21))])
def test_an_output_tensor_that_starts_between_two_sectors(dim, sides):
    """Outputs 16 bytes past a 32-byte boundary are written in halves: the same bits, and nothing around them."""
    import torch
    import paper_2504_09261_b200 as hb
    heads, batch = 6, 2
    caches = [hb.HackCache(1, heads, dim, batch, sides, hb.HACK_BF16, [0, 1] * (heads // 2), 100, 400) for _ in range(2)]
    g = torch.Generator(device="cuda").manual_seed(dim)
    for k, side in enumerate(sides):
        q, kk, v = (torch.randn((batch, heads, side * side, dim), generator=g, device="cuda").bfloat16() for _ in range(3))
        out = torch.empty_like(q)
        room = torch.full((q.numel() + 16,), 7.0, dtype=torch.bfloat16, device="cuda")
        odd = room[8:-8].view(q.shape)
        assert out.data_ptr() % 32 == 0 and odd.data_ptr() % 32 == 16
        caches[0].hack_scale_step(0, k, q, kk, v, out)
        caches[1].hack_scale_step(0, k, q, kk, v, odd)
        assert torch.equal(out.view(torch.int16), odd.view(torch.int16)), k
        assert bool((room[:8] == 7).all()) and bool((room[-8:] == 7).all())
    for c in caches:
        c.hack_poll_status()
        c.close()


@pytest.mark.parametrize("heads,batch,sides,b_c,b_s", [
    (16, 16, (2, 8, 20, 29), 33, 1045),          # 7 query tiles, contextual heads of one short block: several rounds of one tile
    (30, 8, (3, 9, 18), 128, 396),               # 3 tiles, a whole block and a last block of 12 keys
    (20, 15, (2, 10, 13, 24), 230, 700),         # 5 tiles, more units than half SMs
    (5, 60, (9, 10, 11), 400, 400),              # one tile, nothing is evicted
])
def test_odd_numbers_of_query_tiles_on_half_an_sm(heads, batch, sides, b_c, b_s):
    decode(64, heads, batch, sides, b_c, b_s, [(0, 0), (0, 1), (batch // 2, heads - 1), (batch - 1, heads - 2)])
