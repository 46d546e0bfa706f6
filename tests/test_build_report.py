"""Registers that the kernels were compiled to: a spill in a scoring loop costs 1 to 10 % of a call."""
import os
import re

import pytest

from paper_2502_00299_b200 import build


def _spills(src):
    """kernel name -> bytes of spill stores"""
    build.build()
    path = build.report_path(src)
    if not os.path.exists(path):
        pytest.skip("the library came built without its reports")
    out, name = {}, None
    for line in open(path):
        m = re.search(r"Compiling entry function '(\S+)'", line)
        name = m.group(1) if m else name
        m = re.search(r"(\d+) bytes spill stores", line)
        if m and name:
            out[name] = int(m.group(1))
    return out


def test_layer_kernels_do_not_spill():
    spills = _spills("layer_resident.cu")
    assert sum("layer_resident_kernel" in k for k in spills) == 36 and not any(spills.values()), spills


# (two query tiles, or a ring that continues in scratch; the selection's longer bodies would spill here too)
@pytest.mark.parametrize("c,limit", [(5, 6), (8, 28), (10, 0), (16, 4), (20, 0), (32, 48)])
def test_big_model_kernels_spill_no_more_than_their_epilogue_has_to(c, limit):
    found = [v for k, v in _spills("model_kernel.cu").items() if f"model_kernelILi{c}ELb1E" in k]
    assert len(found) == 1 and found[0] <= limit, found
