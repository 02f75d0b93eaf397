"""The compression launch at sizes for which its dispatch rule has different shapes to choose from: more
heads than SMs (two CTAs per SM), candidate lists past the accumulators in tensor memory (bounce accumulators,
logits in shared memory or formed again), few heads of long lists (clusters), and a select that has to settle
ties in its last digit.  That the compression launch is the one that runs is asserted (the last step is two launches);
which shape the rule, a time model, takes for it is not visible from here.
Oracle and bars are those of the parity tests."""
from dataclasses import replace

import numpy as np
import pytest

from workloads import get_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("base,heads,batch,sides,b_c,b_s,policy", [
    (1, 20, 16, (1, 2, 5, 9, 13, 16), 68, 400, 0),          # 320 heads of up to 6 chunks
    (3, 30, 8, (1, 3, 7, 12, 19), 130, 257, 1),             # the same at head_dim 128, current scale competes
    (1, 15, 12, (1, 4, 9, 25, 41), 700, 1300, 0),           # 180 heads, lists past the accumulators of one CTA
    (3, 30, 5, (1, 4, 13, 29, 37), 900, 2100, 0),           # the same at head_dim 128: logits formed a second time
    (3, 3, 1, (1, 4, 11, 17, 30), 257, 640, 1),             # 3 heads: large clusters, ragged last chunks
])
def test_launch_shapes(base, heads, batch, sides, b_c, b_s, policy):
    from parity_util import run_parity
    cfg = replace(get_config(base, n_layers=1), name=f"shape-{heads}x{batch}", n_heads=heads, batch=batch, sides=sides,
                  budget_c=b_c, budget_s=b_s)
    rep = run_parity(cfg, [0], fused=True, heads_per_layer=6, policy=policy, gen_on_gpu=True)
    assert rep.ok(), rep.problems[:5]
    assert rep.compressed_heads > 0
    assert rep.evicting_launches[-1] == 2, rep.evicting_launches


@pytest.mark.parametrize("head_dim,heads", [(64, 2), (128, 200)])
def test_equal_scores_keep_the_lowest_indices(head_dim, heads):
    """All keys zero: every score is the same, so all three digits are needed and the survivors are the
    lowest candidate indices (contextual heads) or those behind the protected ones (structural heads)."""
    import torch
    import paper_2504_09261_b200 as hb
    sides, b_c, b_s = (2, 3, 20, 30), 301, 1201
    mask = np.array([[h % 2 for h in range(heads)]], dtype=np.uint8)
    cache = hb.HackCache(1, heads, head_dim, 1, sides, hb.HACK_BF16, mask, b_c, b_s)
    for k, side in enumerate(sides):
        z = torch.zeros((1, heads, side * side, head_dim), dtype=torch.bfloat16, device="cuda")
        cache.hack_scale_step(0, k, torch.randn_like(z), z, z, torch.empty_like(z))
    for h in (0, 1, heads - 2, heads - 1):
        pos = np.frombuffer(cache.hack_read_head(0, 0, h, 2), dtype=np.int32)
        stored = 13 + 400
        want = np.arange(b_c) if mask[0, h] else np.concatenate([np.arange(b_s - 900), np.arange(stored, stored + 900)])
        assert np.array_equal(pos, want)
    cache.close()
