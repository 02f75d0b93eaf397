"""The fp32 kernels at the edges of their tiles, against fp64 evaluations of the same definitions.

Attention bar 1e-5 max-abs, the one the parity tests hold fp32 outputs to: inputs are N(0, 1), so a
logit is a sum of at most 128 products with |q . k| * scale below about 6; its rounding error is at
most 128 * 2^-24 * 6 / 6 = 8e-6 in the worst case and about sqrt(128) * 2^-24 = 7e-7 as it comes, it
enters the output relatively, and |O| is of the order of 1 and below 5."""
import math

import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()


@pytest.mark.parametrize("head_dim", [64, 128])
@pytest.mark.parametrize("sides", [(1,), (4, 4), (4, 4, 1), (5, 6), (1, 8, 8), (3, 11)])
def test_fp32_attention_over_ragged_tiles(sides, head_dim):
    """Lengths of 1, 32, 33, 61, 129 and 130 keys: one key, exact tiles, one key more, key groups
    without a tile; 1 to 121 queries; staged and fused calls."""
    import numpy as np
    import torch
    import paper_2504_09261_b200 as hb
    heads, batch, total = 3, 2, sum(s * s for s in sides)
    mask = np.array([[1, 0, 1]], dtype=np.uint8)
    g = torch.Generator(device="cuda").manual_seed(total + head_dim)
    caches = [hb.HackCache(1, heads, head_dim, batch, sides, hb.HACK_F32, mask, total, total,
                            n_init_scales=1) for _ in range(2)]
    ks, vs = [], []
    for k, side in enumerate(sides):
        q, kk, v = (torch.randn((batch, heads, side * side, head_dim), generator=g, device="cuda") for _ in range(3))
        ks.append(kk.double())
        vs.append(v.double())
        fused, staged = torch.full_like(q, float("nan")), torch.full_like(q, float("nan"))
        caches[0].hack_scale_step(0, k, q, kk, v, fused)
        scores = torch.zeros((batch * heads, caches[1].cand_stride), device="cuda")
        idx = torch.zeros((batch * heads, caches[1].kept_stride), dtype=torch.int32, device="cuda")
        caches[1].hack_score(0, k, q, kk, scores)
        caches[1].hack_select(0, k, scores, idx)
        caches[1].hack_compact(0, k, idx, kk, v)
        caches[1].hack_attend(0, k, q, staged)
        z = q.double() @ torch.cat(ks, 2).transpose(2, 3) / math.sqrt(head_dim)
        ref = z.softmax(-1) @ torch.cat(vs, 2)
        assert (fused.double() - ref).abs().max() <= 1e-5
        assert (staged.double() - ref).abs().max() <= 1e-5
    for c in caches:
        c.close()


@pytest.mark.parametrize("dtype", ["f32", "bf16"])
@pytest.mark.parametrize("n_cand,n_obs,head_dim", [(1, 1, 64), (127, 8, 128), (128, 31, 64), (129, 32, 128), (1153, 32, 64),
                                                   (1100, 17, 128), (3000, 32, 64), (4096, 32, 128), (4097, 32, 128)])
def test_dense_scores_over_ragged_chunks(n_cand, n_obs, head_dim, dtype):
    """Chunks of 128 keys cut short, filled and exceeded by one; one, two and four chunks per CTA of a
    cluster, clusters with idle CTAs, and the first size past one launch; observation rows that leave
    warps idle.  Bar as in the parity tests of the scores: 1e-4 relative + 1e-7 (fp32 sums of at most
    4097 terms)."""
    import torch
    import paper_2504_09261_b200 as hb
    rows, n_q = 3, 50
    g = torch.Generator(device="cuda").manual_seed(n_cand)
    dt = torch.float32 if dtype == "f32" else torch.bfloat16
    q = torch.randn((rows, n_q, head_dim), generator=g, device="cuda").to(dt)
    k = torch.randn((rows, n_cand, head_dim), generator=g, device="cuda").to(dt)
    scores = torch.full((rows, n_cand + 3), -1.0, device="cuda")
    hb.hack_score_noalloc(q, k, scores, rows, n_q, n_cand, n_cand + 3, head_dim,
                          hb.HACK_F32 if dtype == "f32" else hb.HACK_BF16, n_obs)
    obs = [m * n_q // n_obs for m in range(n_obs)]
    z = torch.einsum("rnd,rcd->rnc", q[:, obs].double(), k.double()) / math.sqrt(head_dim)
    ref = z.softmax(-1).sum(1)
    got = scores[:, :n_cand].double()
    assert bool(((got - ref).abs() <= 1e-4 * torch.maximum(got.abs(), ref.abs()) + 1e-7).all())
    assert bool((scores[:, n_cand:] == -1.0).all())


@pytest.mark.parametrize("head_dim,b_c,b_s,policy", [(64, 255, 257, 1), (64, 256, 512, 0), (128, 127, 129, 1), (128, 1, 383, 0)])
def test_selection_that_moves_the_rows(head_dim, b_c, b_s, policy):
    """fp32 steps small enough for selection and compaction in one launch, kept lengths around the rows of
    its rounds (256 at head_dim 64, 128 at 128), against the oracle and the separate launches."""
    from dataclasses import replace
    from parity_util import run_parity
    from workloads import get_config
    cfg = replace(get_config(0), name=f"select-move-{head_dim}", n_heads=4, batch=2, head_dim=head_dim, sides=(1, 3, 9, 13, 17),
                  budget_c=b_c, budget_s=b_s)
    rep = run_parity(cfg, [0], fused=True, policy=policy)
    assert rep.ok(), rep.problems[:5]
    assert rep.compressed_heads > 0
    assert rep.evicting_launches[-1] == 3, rep.evicting_launches      # scores, selection with the moves, attention


@pytest.mark.parametrize("head_dim,heads,batch,sides,b_c,b_s", [
    (64, 16, 2, (2, 7, 18), 40, 377), (64, 13, 3, (3, 11, 17, 19), 33, 800), (128, 16, 1, (2, 9, 18, 21), 130, 850),
    (128, 20, 1, (1, 16, 17), 545, 546), (128, 11, 2, (2, 23, 24), 1, 1000),
])
def test_query_tiles_that_ctas_share(head_dim, heads, batch, sides, b_c, b_s):
    """More query tiles than SMs, heads of one and of two lengths: shares that begin and end inside a tile, in its
    last round, and tiles of one round.  Against fp64 attention over the rows the cache reports."""
    import numpy as np
    import torch
    import paper_2504_09261_b200 as hb
    mask = (np.arange(heads) % 2).astype(np.uint8)[None]
    cache = hb.HackCache(1, heads, head_dim, batch, sides, hb.HACK_F32, mask, b_c, b_s)
    g = torch.Generator(device="cuda").manual_seed(heads * batch)
    for _ in range(2):                                   # the second time on counters the first has left behind
        cache.hack_reset()
        ks, vs = [], []
        for k, side in enumerate(sides):
            q, kk, v = (torch.randn((batch, heads, side * side, head_dim), generator=g, device="cuda") for _ in range(3))
            ks.append(kk)
            vs.append(v)
            out = torch.full_like(q, float("nan"))
            cache.hack_scale_step(0, k, q, kk, v, out)
            kc, vc = torch.cat(ks, 2).double(), torch.cat(vs, 2).double()
            for b in range(batch):
                for h in range(heads):
                    pos = torch.from_numpy(np.frombuffer(cache.hack_read_head(0, b, h, 2), dtype=np.int32).copy()).long().cuda()
                    z = q[b, h].double() @ kc[b, h, pos].T / math.sqrt(head_dim)
                    ref = z.softmax(-1) @ vc[b, h, pos]
                    assert (out[b, h].double() - ref).abs().max() <= 1e-5, (k, b, h)
    cache.close()


@pytest.mark.parametrize("heads,batch,sides", [(16, 1, (2, 24, 18)), (13, 2, (5, 22, 19))])
def test_query_tiles_that_ctas_share_at_head_dim_64(heads, batch, sides):
    """Sizes that head_dim 64 serves in shares: 176 tiles of 8 rounds, 312 of 7."""
    total = sum(s * s for s in sides)
    test_query_tiles_that_ctas_share(64, heads, batch, sides, total, total)


@pytest.mark.parametrize("head_dim,heads", [(128, 33), (128, 36), (128, 80), (64, 9), (64, 40)])
def test_selection_that_moves_the_rows_in_clusters_of_every_size(head_dim, heads):
    """Four, two and one CTA per head at head_dim 128; at head_dim 64 as many as leave the attention its SMs."""
    from dataclasses import replace
    from parity_util import run_parity
    from workloads import get_config
    cfg = replace(get_config(0), name=f"select-move-{head_dim}-{heads}", n_heads=heads, batch=1, head_dim=head_dim, sides=(1, 3, 9, 13, 17),
                  budget_c=150, budget_s=380)
    rep = run_parity(cfg, [0], fused=True, heads_per_layer=6, policy=1)
    assert rep.ok(), rep.problems[:5]
    assert rep.evicting_launches[-1] <= 4, rep.evicting_launches      # scores in one or two launches, selection with the moves, attention
