"""Steps that merge through hack_scale_step, whose compression launch lists what contextual heads keep and discard and
moves the rows of the structural ones: stored rows, positions and outputs equal those of the stage calls bit for bit, for both
head sizes, structural heads that keep the new scale, let it compete or evict nothing, and lists that one CTA has to
look through twice."""
from dataclasses import replace

import pytest

from workloads import SyntheticQKV, get_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("base", [1, 3], ids=["head_dim_64", "head_dim_128"])
@pytest.mark.parametrize("sides,budget_c,budget_s,policy,heads,batch", [
    ((1, 2, 4, 7, 12, 20), 300, 500, 0, 5, 2),       # the new scale is protected
    ((1, 2, 4, 7, 12, 20), 300, 500, 1, 5, 2),       # it competes
    ((1, 2, 4, 7, 12, 20), 300, 614, 0, 4, 3),       # structural heads evict nothing
    ((1, 2, 4, 7, 12, 20), 1, 600, 1, 3, 1),         # all but one entry are discarded
    ((1, 2, 4, 7, 12, 66), 130, 4300, 1, 40, 2),     # 37 chunks of keys in one or two CTAs per head
])
def test_fused_and_staged_steps_merge_alike(base, sides, budget_c, budget_s, policy, heads, batch):
    import torch
    import paper_2504_09261_b200 as hb
    cfg = replace(get_config(base, n_layers=1), name="merge-fused", n_heads=heads, batch=batch, sides=sides)
    dev = torch.device("cuda:0")
    gen = SyntheticQKV(cfg, device=dev)
    mask = gen.head_is_contextual.cpu().numpy()
    assert 0 < mask.sum() < heads
    staged, fused = (hb.HackCache(1, heads, cfg.head_dim, batch, cfg.sides, hb.HACK_BF16, mask, budget_c, budget_s, merge_last=True,
                                  overflow_policy=policy) for _ in range(2))
    scores = torch.empty((batch * heads, staged.cand_stride), dtype=torch.float32, device=dev)
    idx = torch.empty((batch * heads, staged.kept_stride), dtype=torch.int32, device=dev)
    for k in range(cfg.n_scales):
        q, kk, v = (t.to(dev) for t in gen.qkv(0, k))
        info = staged.hack_step_info(0, k)
        outs = [torch.full_like(q, float("nan")) for _ in range(2)]
        staged.hack_score(0, k, q, kk, scores)
        staged.hack_select(0, k, scores, idx)
        staged.hack_compact(0, k, idx, kk, v)
        staged.hack_attend(0, k, q, outs[0])
        before = fused.hack_launch_count()
        fused.hack_scale_step(0, k, q, kk, v, outs[1])
        launches = fused.hack_launch_count() - before
    # (scales before the last may be one launch, whose probabilities carry more bits than the stage calls')
    assert torch.equal(outs[0].view(torch.int16), outs[1].view(torch.int16))
    assert info.triggered_c and bool(info.triggered_s) == (budget_s < info.cand_s)
    assert launches == 7, launches               # lists, scratch copies, move, copy, counterparts, averages, attention
    assert staged.hack_get_lengths(0) == fused.hack_get_lengths(0)
    for b in range(batch):
        for h in range(min(heads, 8)):
            for which in (0, 1, 2):
                assert staged.hack_read_head(0, b, h, which) == fused.hack_read_head(0, b, h, which), (b, h, which)
    for c in (staged, fused):
        c.hack_poll_status()
        c.close()
