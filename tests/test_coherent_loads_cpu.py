"""Step kernels are resident while their predecessor still writes (programmatic
stream serialization), so nothing that a step kernel writes may be read through
the non-coherent path: only twiddle tables and descriptors are."""
import os
import re

import pytest

from paper_0710_5912_gb300 import _native

READ_ONLY = {"tw", "twff", "descs"}
SOURCES = sorted(f for f in os.listdir(_native.CSRC) if f.startswith("step_"))


@pytest.mark.parametrize("name", SOURCES)
def test_step_kernels_read_what_they_write_with_plain_loads(name):
    with open(os.path.join(_native.CSRC, name)) as f:
        code = re.sub(r"//.*", "", f.read())
    assert set(re.findall(r"__ldg\(\s*(\w+)", code)) <= READ_ONLY
    assert len(re.findall(r"__ldg\b", code)) == len(re.findall(r"__ldg\(\s*\w+", code))
    assert set(re.findall(r"__restrict__\s+(\w+)", code)) <= READ_ONLY
    assert "ld.global.nc" not in code
