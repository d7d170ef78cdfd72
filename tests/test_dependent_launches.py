"""Kernels that may be resident while the kernel ahead of them still writes
their inputs (programmatic dependent launches) must not read those through the
read-only path: it is defined only for memory that nothing writes during the
kernel's whole life, and such loads may move above the wait."""
import os
import re

import pytest

from paper_2510_01764_gb300 import build


@pytest.mark.parametrize("src", [s for s in os.listdir(build.CSRC) if s.endswith((".cu", ".h"))])
def test_no_read_only_loads(src):
    with open(os.path.join(build.CSRC, src)) as f:
        code = re.sub(r"//[^\n]*|/\*.*?\*/", "", f.read(), flags=re.S)
    assert not re.search(r"\b__ldg\b|ld\.global\.nc|\b__restrict__\b", code)
