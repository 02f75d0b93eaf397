"""Small steps in one launch of more heads than clusters of the size that would spread them best find a place (46 of 3
CTAs, 35 of 4, 24 of 6 on 148 SMs), and compression of as many heads as clusters of an odd size would just find places for (45 of 3 CTAs, 26 of 5, 15 of 7 on
148 SMs) and of one more than they may take: the cluster size changes there.  Protocol and bars are those of the parity tests."""
from dataclasses import replace

import pytest

from workloads import get_config

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("base,heads", [(1, 42), (1, 43), (3, 45), (3, 24), (1, 26), (3, 15)])
def test_heads_at_the_line_of_a_cluster_size(base, heads):
    from parity_util import run_parity
    cfg = replace(get_config(base, n_layers=1), name=f"places-{heads}", n_heads=heads, batch=1, sides=(1, 2, 5, 9, 14, 23),
                  budget_c=260, budget_s=520)
    rep = run_parity(cfg, [0], fused=True, heads_per_layer=4, policy=1, gen_on_gpu=True)
    assert rep.ok(), rep.problems[:5]
    assert rep.compressed_heads > 0


@pytest.mark.parametrize("dtype", ["bf16", "fp32"])
@pytest.mark.parametrize("head_dim,heads", [(128, 45), (128, 46), (64, 35), (128, 35), (64, 24), (128, 23)])
def test_heads_at_the_places_of_small_clusters(head_dim, heads, dtype):
    from parity_util import run_parity
    base = get_config(0) if dtype == "fp32" else get_config(3 if head_dim == 128 else 1, n_layers=1)
    cfg = replace(base, name=f"small-{heads}", n_heads=heads, batch=1, head_dim=head_dim, sides=(1, 2, 3, 5, 7, 9, 11),
                  budget_c=60, budget_s=100)
    rep = run_parity(cfg, [0], fused=True, heads_per_layer=4, policy=1)
    assert rep.ok(), rep.problems[:5]
    assert rep.compressed_heads > 0


@pytest.mark.parametrize("dtype,head_dim,heads,sides,b_c,b_s", [
    ("bf16", 128, 46, (1, 2, 5, 12), 20, 166), ("fp32", 64, 24, (1, 2, 4, 7, 13), 24, 231), ("fp32", 128, 36, (1, 2, 4, 10), 18, 113),
])
def test_contextual_heads_that_wait_for_the_first_clusters(dtype, head_dim, heads, sides, b_c, b_s):
    """One launch whose last clusters, contextual heads of few keys, start when the first ones have ended."""
    from parity_util import run_parity
    base = get_config(0) if dtype == "fp32" else get_config(3 if head_dim == 128 else 1, n_layers=1)
    cfg = replace(base, name=f"waiting-{heads}", n_heads=heads, batch=1, head_dim=head_dim, sides=sides, budget_c=b_c, budget_s=b_s)
    rep = run_parity(cfg, [0], fused=True, heads_per_layer=8, policy=1)
    assert rep.ok(), rep.problems[:5]
    assert rep.evicting_launches[-1] == 1, rep.evicting_launches
