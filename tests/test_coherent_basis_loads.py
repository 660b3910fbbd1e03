"""Kernels that write basis columns and read them back in the same launch (the batched solver, the
single-launch restart cycle) must not read them through the non-coherent path: ld.global.nc is
defined only for data that nothing writes while the kernel runs."""
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2009_12101_gb300", "csrc")


def _code(name):
    with open(os.path.join(CSRC, name)) as f:
        return re.sub(r"//[^\n]*", "", f.read())


@pytest.mark.parametrize("name", ["cbg_batched.cuh", "cbg_cycle.cuh"])
def test_basis_is_read_coherently(name):
    text = _code(name)
    assert "encode_store" in text                      # these write codes
    assert "ldg_stream" not in text and ".nc" not in text
    # __ldg (the same path) only on the operator: structure, values, chunk offsets
    for arg in re.findall(r"__ldg\(([^;]*?)\)", text):
        assert re.match(r"(a\.(prow|pcol|pvals|rowptr|col|valdf|sell_col|sell_val64)|off|vhp|vlp|vlo)\b", arg), arg
