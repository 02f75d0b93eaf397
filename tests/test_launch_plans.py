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
    cl = plans.move_ctas(heads, out[2] if dim == 64 else 0)
    best = min(t for t in us if t is not None)
    assert us[{1: 0, 2: 1, 4: 2}[cl]] <= 1.02 * best, (cl, list(out))
