"""Register use of kernels whose registers are the limit of their CTAs per SM, from what the compiler reports: forms that
must not spill."""
import os
import re
import subprocess

import pytest

from paper_2504_09261_b200 import build

SPILL = re.compile(r"Function properties for (\S+)\s+\d+ bytes stack frame, (\d+) bytes spill stores, (\d+) bytes spill loads")


def spills(source):
    res = subprocess.run([build._nvcc()] + build.NVCC_FLAGS + ["-Xptxas", "-v", "-c", os.path.join(build.CSRC, source), "-o", os.devnull],
                         capture_output=True, text=True)
    assert res.returncode == 0, res.stderr
    return {name: (int(st), int(ld)) for name, st, ld in SPILL.findall(res.stderr)}


# template arguments as they stand in the mangled name: <head_dim, form>
@pytest.mark.parametrize("source,kernel,forms", [
    ("attend_simt.cu", "attend_simt_kernel", ["ILi64ELi0EE", "ILi64ELi1EE", "ILi128ELi0EE", "ILi128ELi1EE", "ILi128ELi2EE"]),
])
def test_no_spills(source, kernel, forms):
    found = spills(source)
    for form in forms:
        mine = [v for name, v in found.items() if kernel + form in name]
        assert mine == [(0, 0)], (form, mine)
