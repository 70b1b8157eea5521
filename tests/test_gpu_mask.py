"""The mask kernel: it keeps no registers in memory, in either argument form."""

import re
from pathlib import Path

import pytest


def test_the_mask_kernel_does_not_spill():
    log = Path(__file__).resolve().parents[1] / "paper_2210_06158_gb300" / "_lib" / "obj" / "trace.ptxas.txt"
    if not log.exists():
        pytest.skip("the library has not been built here")
    found = re.findall(r"Compiling entry function '(\S*k_mask_compact\S*)'.*?(\d+) bytes spill stores, (\d+) bytes spill loads",
                       log.read_text(), re.S)
    assert len(found) == 2
    assert not [f for f in found if int(f[1]) or int(f[2])], found
