"""A recorded DRAM traffic figure counts while the hash of its kernel's sources matches: the list of
sources must hold every header that they include (bench.py, KERNEL_SOURCES)."""
import os
import re

import pytest

import bench
from paper_2601_16911_gb300 import build as B


def included(name):
    with open(os.path.join(B.CSRC, name)) as f:
        return [x for x in re.findall(r'#include\s+"([^"/]+)"', f.read()) if os.path.exists(os.path.join(B.CSRC, x))]


@pytest.mark.parametrize("key", sorted(bench.KERNEL_SOURCES))
def test_kernel_sources_hold_every_included_header(key):
    listed = bench.KERNEL_SOURCES[key]
    missing = sorted({h for f in listed for h in included(f)} - set(listed))
    assert not missing, missing
