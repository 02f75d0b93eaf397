"""A bounded device-side wait that runs out.

Every mbarrier wait in the tensor-core kernels has a limit; when it expires the CTA raises the status
word, drains the copies and MMAs it has in flight, frees its tensor memory and returns.  The limit
is normally about a second, so nothing ever reaches it.  Here hack_set_wait_limit makes it one cycle
for one scoring launch: the consumers' first wait for an accumulator (which needs a key tile from
HBM and an MMA, a microsecond at least) gives up, hack_poll_status reports the time-out, and the
same cache, reset and back on the default limit, then passes the ordinary parity run.  Nothing
spins and nothing faults: the wait itself returns.  The same with whole steps that evict, append or
merge, and a limit that launches behind one another and long units of work must not run into.
"""
from dataclasses import replace

import pytest
import torch

from workloads import SyntheticQKV, get_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("head_dim", [64, 128])
def test_scoring_wait_runs_out_and_the_cache_stays_usable(head_dim):
    import paper_2504_09261_b200 as hb
    from tests.parity_util import make_cache, run_parity
    base = get_config(1 if head_dim == 64 else 3, n_layers=1)
    cfg = replace(base, name=base.name + "-tiny", n_heads=4, batch=1, sides=(1, 2, 4, 8, 12),
                  budget_c=40, budget_s=120)
    gen = SyntheticQKV(cfg)
    mask = gen.head_is_contextual.numpy()
    cache = make_cache(cfg, mask)
    dev = torch.device("cuda:0")
    bh = cfg.batch * cfg.n_heads
    scores = torch.zeros((bh, cache.cand_stride), dtype=torch.float32, device=dev)
    # walk to the first step that scores
    k = 0
    while True:
        info = cache.hack_step_info(0, k)
        q, kk, v = (t.to(dev) for t in gen.qkv(0, k))
        if info.triggered_c or info.triggered_s:
            break
        cache.hack_scale_step(0, k, q, kk, v, torch.empty_like(q))
        k += 1
    cache.hack_poll_status()                       # nothing has gone wrong so far
    with pytest.raises(hb.HackError) as e:
        cache.hack_set_wait_limit(-1)
    assert e.value.status == 1
    cache.hack_set_wait_limit(1)
    cache.hack_score(0, k, q, kk, scores)
    with pytest.raises(hb.HackError) as e:
        cache.hack_poll_status()
    assert e.value.status == 6, str(e.value)          # HACK_ERR_TIMEOUT
    cache.hack_poll_status()                       # the word was cleared by the call that reported it
    cache.hack_set_wait_limit(0)
    # the context, the library and this very cache are as usable as before
    rep = run_parity(cfg, layers=[0], fused=True, staged_cache=cache)
    assert rep.ok(), rep.summary() + "\n" + "\n".join(rep.problems)
    assert rep.compressed_heads > 0
    cache.close()


def _aborted_last_step(head_dim, sides, budget_c, budget_s, heads=6, batch=1, merge=False):
    """A decode whose last step runs with a limit of one cycle; then a clean decode on the same cache and
    on a fresh one, whose rows, positions and outputs have to be the same."""
    import numpy as np
    import paper_2504_09261_b200 as hb
    mask = (np.arange(heads) % 2).astype(np.uint8)[None]
    dev = torch.device("cuda:0")
    g = torch.Generator(device=dev).manual_seed(head_dim + len(sides))
    steps = [tuple(torch.randn((batch, heads, s * s, head_dim), generator=g, device=dev).bfloat16() for _ in range(3)) for s in sides]
    caches = [hb.HackCache(1, heads, head_dim, batch, sides, hb.HACK_BF16, mask, budget_c, budget_s, merge_last=merge) for _ in range(2)]

    def decode(cache, last_limit=0):
        cache.hack_reset()
        for k, (q, kk, v) in enumerate(steps):
            if k == len(steps) - 1:
                cache.hack_poll_status()
                cache.hack_set_wait_limit(last_limit)
            out = torch.full_like(q, float("nan"))
            cache.hack_scale_step(0, k, q, kk, v, out)
        return out

    decode(caches[0], 1)
    status = 0
    try:
        caches[0].hack_poll_status()
    except hb.HackError as e:
        status = e.status
    caches[0].hack_set_wait_limit(0)
    outs = [decode(c) for c in caches]
    for c in caches:
        c.hack_poll_status()
    assert torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))
    for h in range(heads):
        for which in (0, 1, 2):
            assert caches[0].hack_read_head(0, batch - 1, h, which) == caches[1].hack_read_head(0, batch - 1, h, which)
    for c in caches:
        c.close()
    return status


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("sides,budget_c,budget_s", [
    ((1, 2, 4, 12, 26), 300, 760),      # both types evict; at head_dim 64 two CTAs of the attention share an SM
    ((1, 2, 14, 24, 40), 2000, 2300),   # the same where a CTA takes two query tiles
    ((1, 2, 4, 12, 26), 300, 2000),     # structural heads append beside the compression of the others
    ((1, 2, 6, 12, 22), 300, 600),      # lists of few blocks
])
def test_a_step_that_evicts_gives_up_and_the_cache_stays_usable(head_dim, sides, budget_c, budget_s):
    assert _aborted_last_step(head_dim, sides, budget_c, budget_s) == 6    # HACK_ERR_TIMEOUT


@pytest.mark.parametrize("head_dim,sides", [(64, (1, 2, 20)), (64, (1, 20, 40)), (128, (1, 20, 40))])
def test_an_appending_step_with_a_short_limit(head_dim, sides):
    """The attention blocks in its waits for a while before it looks at the clock, so that it may well get through."""
    assert _aborted_last_step(head_dim, sides, 4000, 4000, heads=40) in (0, 6)


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("budget_s", [760, 2000])
def test_a_merging_step_that_gives_up_reads_rows_of_its_heads_only(head_dim, budget_s):
    """Its lists of kept and discarded rows are not formed then, and the launches behind read rows through them."""
    assert _aborted_last_step(head_dim, (1, 2, 4, 12, 26), 300, budget_s, merge=True) == 6


def test_the_limit_counts_neither_the_launch_ahead_nor_whole_units_of_work():
    """Two attention launches of three rounds of CTAs, back to back: a CTA of the second one waits for the first for as
    long as that launch's last CTAs take, and a unit is 83 blocks of 128 keys, 130 us.  The limit lies below either, at
    about 40 us, far above what a wait inside the loop takes (a block is 1.6 us)."""
    import paper_2504_09261_b200 as hb
    dev = torch.device("cuda:0")
    sides, heads, batch, dim = (1, 2, 80, 64), 16, 2, 128
    cache = hb.HackCache(2, heads, dim, batch, sides, hb.HACK_BF16, [0, 1] * heads, 20000, 20000)
    g = torch.Generator(device=dev).manual_seed(5)
    steps = [tuple(torch.randn((batch, heads, s * s, dim), generator=g, device=dev).bfloat16() for _ in range(3)) for s in sides]
    outs = [torch.empty_like(steps[-1][0]) for _ in range(4)]
    for limit in (0, 75000):
        cache.hack_reset()
        for k, (q, kk, v) in enumerate(steps):
            cache.hack_set_wait_limit(limit if k == len(steps) - 1 else 0)
            for layer in range(2):
                cache.hack_scale_step(layer, k, q, kk, v, outs[layer + (2 if limit else 0)] if k == len(steps) - 1 else torch.empty_like(q))
        cache.hack_poll_status()                   # raises if a wait ran out
    assert torch.equal(outs[0].view(torch.int16), outs[2].view(torch.int16))
    assert torch.equal(outs[1].view(torch.int16), outs[3].view(torch.int16))
    cache.close()
