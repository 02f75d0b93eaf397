"""Merge of the last scale where the lists of discarded entries are long: more entries than a block of the averaging
kernel sifts at a time (4 096), more of them per warp than it lists before it works them off (256), and a last block with
two retained rows.  Protocol and bar are those of the merge's parity test."""
import pytest

from test_gpu_merge import _built, test_merge_matches_the_oracle as _check  # noqa: F401

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("base", [1, 3], ids=["head_dim_64", "head_dim_128"])
def test_lists_longer_than_a_block_sifts(base):
    _check(base, (1, 2, 4, 7, 12, 66), 130, 4700)
