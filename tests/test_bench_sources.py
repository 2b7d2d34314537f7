"""A recorded traffic figure counts only while the profiled kernel's sources are unchanged, so every file that the
kernel is built from has to be among them."""
import os
import re

import pytest

import bench


def _built_from(name, seen):
    seen.add(name)
    with open(os.path.join(bench.CSRC, name)) as f:
        for inc in re.findall(r'^#include "([^"]+)"', f.read(), re.M):
            if inc not in seen and os.path.exists(os.path.join(bench.CSRC, inc)):
                _built_from(inc, seen)
    return seen


@pytest.mark.parametrize("kernel", sorted(bench.KERNEL_SOURCES))
def test_every_file_a_kernel_is_built_from_counts(kernel):
    listed = bench.KERNEL_SOURCES[kernel]
    assert set(listed) == _built_from(listed[0], set())
