"""A whole decode enqueued on one stream without synchronising, the way a model drives the library: one set of
Q, K, V and output buffers per scale serves every layer, copies on the same stream fill it before a step and
take the result away behind it.

The attention launch of a step starts while the compression launch ahead of it still runs, reads the
caller's tensors ahead of its dependency wait and, for heads that evict nothing, also writes the output and the
cache early.  If that reached past the copies ahead of the step, or if a launch of a later step or a copy started before
everything of this one had been read, results would change.  They are compared byte for byte with the same
decode on tensors of its own per step, synchronised after each."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LAYERS = 5


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("dtype,dim,heads,batch,sides,b_c,b_s,policy", [
    # tensor-core attention behind the compression: contextual heads evict alone, then beside protected structural ones
    ("bf16", 128, 16, 2, (1, 2, 4, 8, 12, 20, 26, 32), 500, 1200, 0),
    ("bf16", 128, 7, 3, (1, 3, 7, 15, 27, 37), 475, 951, 1),            # both evict, the new scale competes
    ("bf16", 64, 30, 8, (1, 2, 4, 9, 13, 18, 24), 112, 700, 0),         # one query tile on half an SM, two compression CTAs per SM
    ("bf16", 64, 6, 1, (1, 2, 12, 30, 5, 4), 500, 2000, 0),             # mma attention behind the compression, one type evicts
    ("bf16", 64, 6, 2, (1, 2, 12, 30, 5, 4), 500, 910, 0),              # ... and protected structural heads
    ("bf16", 64, 16, 1, (1, 2, 3, 4, 5, 6, 8, 10, 13, 16), 68, 612, 0),  # small steps in one launch
    ("f32", 64, 16, 1, (1, 2, 3, 4, 5, 6, 8, 10, 13, 16), 34, 374, 0),
    ("f32", 128, 5, 2, (1, 2, 5, 9, 16, 21), 90, 400, 1),               # separate fp32 launches
])
def test_reused_buffers_without_synchronising(dtype, dim, heads, batch, sides, b_c, b_s, policy):
    import torch
    import paper_2504_09261_b200 as hb
    tdt = torch.float32 if dtype == "f32" else torch.bfloat16
    mask = ((np.arange(LAYERS * heads).reshape(LAYERS, heads) * 7) % 5 < 2).astype(np.uint8)
    caches = [hb.HackCache(LAYERS, heads, dim, batch, sides, hb.HACK_F32 if dtype == "f32" else hb.HACK_BF16, mask, b_c, b_s,
                            overflow_policy=policy) for _ in range(2)]
    g = torch.Generator(device="cuda").manual_seed(dim + heads)
    data = [[tuple(torch.randn((batch, heads, s * s, dim), generator=g, device="cuda").to(tdt) for _ in range(3))
             for _ in range(LAYERS)] for s in sides]
    want = []
    for k in range(len(sides)):
        for l in range(LAYERS):
            out = torch.full_like(data[k][l][0], float("nan"))
            caches[0].hack_scale_step(l, k, *data[k][l], out)
            torch.cuda.synchronize()
            want.append(out)
    sets = [[torch.empty_like(data[k][0][0]) for _ in range(4)] for k in range(len(sides))]
    got = [[torch.empty_like(w) for w in want] for _ in range(2)]
    stream = torch.cuda.Stream()
    stream.wait_stream(torch.cuda.current_stream())
    evicting = 0
    with torch.cuda.stream(stream):
        for turn in got:                                    # the second decode follows the first without a pause
            caches[1].hack_reset()
            i = 0
            for k in range(len(sides)):
                q, kk, v, out = sets[k]
                for l in range(LAYERS):
                    for dst, src in zip((q, kk, v), data[k][l]):
                        dst.copy_(src)
                    info = caches[1].hack_step_info(l, k)
                    evicting += info.triggered_c or info.triggered_s
                    caches[1].hack_scale_step(l, k, q, kk, v, out, stream.cuda_stream)
                    turn[i].copy_(out)
                    i += 1
    torch.cuda.synchronize()
    assert evicting > 0
    for turn in got:
        for i, (x, y) in enumerate(zip(want, turn)):
            assert torch.equal(x.view(torch.uint8), y.view(torch.uint8)), f"scale {i // LAYERS} layer {i % LAYERS}"
    for l in range(LAYERS):
        for b, h in ((0, 0), (batch - 1, heads - 1), (0, heads // 2)):
            for which in (0, 1, 2):
                assert caches[0].hack_read_head(l, b, h, which) == caches[1].hack_read_head(l, b, h, which)
    for c in caches:
        c.hack_poll_status()
        c.close()
