"""Kernels launched programmatically live before the kernel ahead of them has ended,
so they must not read through non-coherent loads, whose data may not change while the
kernel lives and which the compiler may move above the wait: in their files there is
no __ldg and no const __restrict__ pointer but to the plan's integer tables."""
import glob
import os
import re

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2607_16074_gb300", "csrc")
FILES = sorted(f for f in glob.glob(os.path.join(CSRC, "*.cu")))


def _source(path):
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", open(path).read(), flags=re.S)


def _programmatic(src):
    return "pdl_entry();" in src


def test_some_files_launch_programmatically():
    assert sum(_programmatic(_source(f)) for f in FILES) >= 8


@pytest.mark.parametrize("path", FILES, ids=os.path.basename)
def test_programmatic_kernels_read_by_plain_loads(path):
    src = _source(path)
    if not _programmatic(src):
        return
    assert not re.findall(r"__ldg|ld\.global\.nc|__ldcg|__ldca", src)
    const = re.findall(r"const\s+(\w+)\s*\*\s*(?:const\s+)?__restrict__\s*(\w+)", src)
    assert not [c for c in const if c[0] not in ("int", "int32_t")], const
