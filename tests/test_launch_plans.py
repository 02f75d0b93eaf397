"""The host rules that cut launches up (csrc/launch_plans.h), compiled for the CPU: at sizes where both sides were timed
they have to take the faster one.  148 SMs."""
import ctypes
import os
import subprocess

import pytest

from paper_2504_09261_b200 import build

SHIM = """
#include "launch_plans.h"
extern "C" void attention(int dim, int n_new, int kept_s, int kept_c, int heads_s, int heads_c, int* out) {
  const int kept[2] = {kept_s, kept_c}, heads[2] = {heads_s, heads_c};
  const hack::simt::SimtPlan p = hack::simt::simt_plan(dim, n_new, kept, heads, 148);
  out[0] = p.cluster; out[1] = p.shared; out[2] = p.ctas;
}
// clusters of 2, 4 CTAs that 148 SMs take at once
static int places(int ctas) { return ctas == 1 ? 1 << 30 : ctas == 2 ? 74 : 33; }
// the same for the small steps' kernels, whose registers leave room for one or two CTAs on an SM
static int step_places(int ctas, size_t smem, bool two) {
  static const int n[9] = {0, 1 << 29, 74, 45, 33, 26, 22, 18, 16};
  return smem > hack::small_step::kSmemHalf || !two ? n[ctas] : 2 * n[ctas];
}
static size_t smem_bf16(int dim, const hack::small_step::StepShape& s) {
  const size_t kv = (size_t)(s.rows > 128 ? s.rows : 128) * dim * 4;
  return kv + 32 * dim * 2 + (size_t)s.tiles * 16 * dim * 2 + (size_t)s.rows * 12;
}
static size_t smem_f32(int dim, const hack::small_step::StepShape& s) {
  const size_t keys = (size_t)s.rows * (dim + 4) * 4, out = (size_t)8 * 8 * dim * 4;
  return (keys > out ? keys : out) + (size_t)s.rows * dim * 4 + 32 * dim * 4 + (size_t)s.tiles * 8 * dim * 4 + (size_t)s.rows * 28;
}
// 0: two or three launches, else CTAs per head
extern "C" int small_step(int bf16, int dim, int heads_s, int heads_c, int n_new, int cand, int kept_s, int kept_c) {
  using namespace hack::small_step;
  const int heads[2] = {heads_s, heads_c}, cands[2] = {cand, cand}, kept[2] = {kept_s, kept_c}, trig[2] = {1, 1};
  const StepSizes z{dim, n_new, heads, cands, kept, trig, 148};
  StepShape s;
  if (bf16) {
    s.rows = (cand + 15) / 16 * 16;
    return step_shape_bf16(z, s, (n_new + 15) / 16, (cand + 127) / 128, [&](const StepShape& of) { return smem_bf16(dim, of); },
                           [&](int ctas, size_t smem) { return step_places(ctas, smem, dim == 64 && cand <= 512); }) ? s.ctas : 0;
  }
  s.rows = (cand + 3) / 4 * 4;
  return step_shape_f32(z, s, (n_new + 7) / 8, [&](const StepShape& of) { return smem_f32(dim, of); },
                        [&](int ctas, size_t smem) { return step_places(ctas, smem, cand <= 128); }) ? s.ctas : 0;
}
extern "C" int move_ctas(int heads, int attention_ctas) { return hack::move_ctas(heads, attention_ctas, 148, places); }
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    where = tmp_path_factory.mktemp("plans")
    (where / "shim.cpp").write_text(SHIM)
    lib = str(where / "shim.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC, "-I", os.path.join(build.ROOT, "include"),
                    str(where / "shim.cpp"), "-o", lib], check=True)
    return ctypes.CDLL(lib)


# fp32, head_dim 64, keys of one length: query tiles and rounds, us a step in equal shares and with a tile per CTA
@pytest.mark.parametrize("heads,queries,keys,shares,apart", [
    (16, 324, 909, 57.5, 62.5), (16, 676, 2069, 171.1, 188.0), (48, 484, 1393, 238.2, 246.5),
    (37, 324, 909, 103.9, 91.9), (93, 144, 389, 65.2, 60.9), (93, 196, 585, 109.2, 100.4), (93, 324, 909, 221.1, 200.8),
    (93, 676, 2069, 885.5, 831.0), (240, 100, 245, 73.7, 63.7), (128, 81, 145, 33.8, 25.9),
])
def test_query_tiles_in_shares_where_that_is_faster(plans, heads, queries, keys, shares, apart):
    out = (ctypes.c_int * 3)()
    plans.attention(64, queries, keys, keys, heads - heads // 2, heads // 2, out)
    assert out[0] == 1
    assert bool(out[1]) == (shares < apart), list(out)


# lists of two lengths, half of the heads each, behind a compaction
@pytest.mark.parametrize("heads,queries,kept_s,kept_c,shares,apart", [
    (16, 324, 909, 200, 62.7, 79.1), (16, 484, 1300, 200, 98.7, 121.4), (26, 324, 909, 200, 80.1, 88.3), (37, 144, 389, 200, 45.6, 43.3),
    (26, 196, 585, 200, 50.4, 47.9), (16, 324, 344, 35, 41.5, 36.6), (26, 196, 380, 120, 45.1, 39.2), (37, 676, 1300, 200, 190.8, 182.9),
])
def test_query_tiles_in_shares_with_lists_of_two_lengths(plans, heads, queries, kept_s, kept_c, shares, apart):
    out = (ctypes.c_int * 3)()
    plans.attention(64, queries, kept_s, kept_c, heads - heads // 2, heads // 2, out)
    assert bool(out[1]) == (shares < apart), list(out)


# the same at head_dim 128, 10 heads of the longer list and 6 of the other
@pytest.mark.parametrize("queries,kept_s,kept_c,shares,apart", [
    (324, 640, 224, 77, 70), (576, 1216, 224, 138, 170), (1024, 1717, 224, 267, 300),
])
def test_query_tiles_in_shares_at_head_dim_128(plans, queries, kept_s, kept_c, shares, apart):
    out = (ctypes.c_int * 3)()
    plans.attention(128, queries, kept_s, kept_c, 10, 6, out)
    assert bool(out[1]) == (shares < apart), list(out)


# selection with the moves: us a step with 1, 2 and 4 CTAs per head
@pytest.mark.parametrize("dim,heads,queries,kept_s,kept_c,us", [
    (64, 8, 196, 216, 40, (23.0, 23.0, 21.5)), (64, 16, 196, 380, 190, (33.3, 31.7, 36.4)), (64, 16, 256, 276, 40, (28.4, 30.5, 30.0)),
    (64, 26, 196, 216, 40, (28.4, 32.3, 34.3)), (64, 37, 196, 250, 120, (36.9, 36.9, 42.0)), (128, 16, 324, 344, 40, (50.4, 48.1, 45.8)),
    (128, 33, 256, 380, 190, (77.1, 74.0, 70.9)), (128, 37, 144, 250, 120, (47.4, 45.1, 50.0)), (128, 45, 324, 344, 40, (90.5, 88.2, None)),
    (128, 80, 324, 344, 40, (135.0, None, None)), (64, 33, 324, 380, 190, (60.2, 56.3, 55.5)), (64, 45, 256, 380, 190, (57.7, 55.2, None)),
])
def test_ctas_that_move_the_rows_of_a_head(plans, dim, heads, queries, kept_s, kept_c, us):
    out = (ctypes.c_int * 3)()
    plans.attention(dim, queries, kept_s, kept_c, heads - heads // 2, heads // 2, out)
    cl = plans.move_ctas(heads, out[2] if dim == 64 and out[0] == 1 else 0)
    best = min(t for t in us if t is not None)
    assert us[{1: 0, 2: 1, 4: 2}[cl]] <= 1.02 * best, (cl, list(out))


# small steps whose clusters do not all find a place at once, half of the heads of either type, structural heads short of all
# candidates by 8: us a step with the CTAs per head that leave every CTA an SM, with the largest clusters that fit, and in
# launches of their own
@pytest.mark.parametrize("bf16,dim,heads,queries,cand,kept_c,ctas,us", [
    (1, 128, 46, 144, 174, 23, (3, 2), (16.1, 17.9, 17.4)), (1, 128, 46, 144, 174, 43, (3, 2), (17.1, 17.9, 17.7)),
    (1, 128, 46, 144, 174, 87, (3, 2), (19.5, 17.9, 18.9)), (1, 128, 49, 144, 174, 23, (3, 2), (16.6, 17.9, 17.7)),
    (1, 128, 46, 169, 199, 23, (3, 2), (17.2, 18.2, 17.7)), (1, 128, 23, 169, 199, 23, (6, 3), (16.1, 12.5, 16.6)),
    (1, 128, 23, 169, 280, 63, (6, 3), (19.5, 17.1, 17.9)), (1, 128, 34, 121, 151, 23, (4, 2), (15.6, 12.5, 15.6)),
    (1, 128, 46, 81, 111, 23, (3, 2), (14.3, 10.5, 15.1)), (1, 64, 23, 324, 435, 63, (6, 3), (17.9, 20.5, 16.6)),
    (1, 64, 24, 324, 435, 217, (6, 3), (23.3, 20.5, 18.4)), (1, 64, 27, 289, 400, 100, (5, 3), (19.5, 19.7, 17.2)),
    (0, 64, 23, 169, 239, 24, (6, 3), (24.6, 33.3, 32.5)), (0, 64, 23, 169, 311, 24, (6, 3), (26.7, 39.9, 36.9)),
    (0, 64, 23, 169, 311, 103, (6, 3), (35.3, 39.9, 37.4)), (0, 64, 28, 144, 286, 48, (5, 3), (27.9, 37.4, 38.4)),
    (0, 64, 34, 121, 191, 95, (4, 2), (31.5, 28.4, 34.0)), (0, 64, 36, 100, 202, 24, (4, 2), (23.8, 30.2, 33.8)),
    (0, 64, 46, 81, 151, 75, (3, 2), (29.7, 24.8, 31.5)), (0, 128, 34, 121, 142, 18, (4, 2), (35.6, 38.8, 39.7)),
    (0, 128, 36, 100, 121, 18, (4, 2), (30.2, 32.5, 36.2)), (0, 128, 36, 100, 121, 90, (4, 2), (42.6, 32.8, 37.3)),
    (0, 128, 48, 81, 102, 51, (3, 2), (33.3, 28.2, 31.3)), (0, 128, 29, 144, 165, 82, (5, 3), (45.8, 99.0, 36.1)),
    (1, 64, 24, 361, 391, 23, (6, 3), (16.9, 18.7, 16.1)),
])
def test_small_steps_whose_clusters_wait(plans, bf16, dim, heads, queries, cand, kept_c, ctas, us):
    got = plans.small_step(bf16, dim, heads - heads // 2, heads // 2, queries, cand, cand - 8, kept_c)
    assert got in (0,) + ctas, got
    took = us[2] if got == 0 else us[ctas.index(got)]
    assert took <= 1.04 * min(us), (got, us)


def test_a_smaller_cluster_has_to_fit_shared_memory(plans):
    """24 heads x 128, 169 queries, 384 candidates: 6 CTAs of two query tiles fit shared memory, 3 of four do not, and with 6 the last heads
    wait, which two launches (18 to 20 us) are faster than; at 22 heads nobody waits."""
    assert plans.small_step(1, 128, 12, 12, 169, 384, 376, 200) == 0
    assert plans.small_step(1, 128, 11, 11, 169, 384, 376, 200) == 6
