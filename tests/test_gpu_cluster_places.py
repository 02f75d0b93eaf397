"""Compression of as many heads as clusters of an odd size would just find places for (45 of 3 CTAs, 26 of 5, 15 of 7 on
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
