"""The kernels are launched with programmatic dependent launch: one may be resident while the kernel ahead of it
still writes its inputs. Such memory must not be read through the read-only path (``__ldg``, ``ld.global.nc``),
which is defined only where nobody writes while the kernel is resident."""
import glob
import os
import re

import pytest

from paper_2608_03447_gb300 import build

SOURCES = sorted(glob.glob(os.path.join(build.CSRC, "*.cu")) + glob.glob(os.path.join(build.CSRC, "*.cuh")))


def _code(path):
    with open(path) as f:
        text = f.read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", text, flags=re.S)


@pytest.mark.parametrize("path", SOURCES, ids=os.path.basename)
def test_no_read_only_path_load(path):
    code = _code(path)
    found = re.findall(r"__ldg\s*\(|ld\.global(?:\.\w+)*\.nc\b", code)
    assert not found, f"{os.path.basename(path)}: {found}"
