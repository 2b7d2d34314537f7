"""Which row-stage kernel a call gets: the host rule alone, compiled with the host compiler, on both sides of its
lines, for the SM count they were measured on and for half of it."""
import ctypes
import os
import subprocess

import pytest

from paper_2608_03447_gb300 import build

SMALL, STREAM, TMA = 0, 1, 2
KB, MB = 1 << 10, 1 << 20

SHIM = """
#include "asd_dispatch.h"
extern "C" int path_of(int B, int K, int row_bytes, int single, int resident, int fused, int sms) {
  const long long request = static_cast<long long>(K + 1) * row_bytes;
  return static_cast<int>(asd_detail::choose_path(ASD_PATH_AUTO, request * B, request, B, K, single, resident, fused,
                                                  sms));
}
"""


@pytest.fixture(scope="module")
def path_of(tmp_path_factory):
    d = tmp_path_factory.mktemp("dispatch")
    (d / "shim.cpp").write_text(SHIM)
    out = str(d / "shim.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{build.INCLUDE}",
                    f"-I{build.CSRC}", str(d / "shim.cpp"), "-o", out], check=True)
    lib = ctypes.CDLL(out)
    return lambda B, K, row_bytes, single=True, resident=False, fused=False, sms=152: lib.path_of(
        B, K, row_bytes, int(single), int(resident), int(fused), sms)


@pytest.mark.parametrize("sms", [152, 76])
def test_one_cta_requests_of_a_megabyte_up_to_a_cta_per_sm(path_of, sms):
    for K, row in ((8, 6 * KB), (2, 16 * KB)):
        assert path_of(sms, K, row, sms=sms) == SMALL
        assert path_of(sms + 1, K, row, sms=sms) == STREAM


@pytest.mark.parametrize("sms", [152, 76])
@pytest.mark.parametrize("K,row,per_sm", [(0, 34, 11), (4, 200, 3), (8, 200, 2), (31, 8, 1), (0, 1000, 5), (14, 4, 1)])
def test_tiny_requests_as_many_as_fit_at_once(path_of, K, row, per_sm, sms):
    """A CTA of one warp per unit and one for the drafts' logits; 22 warps fit an SM."""
    assert path_of(per_sm * sms, K, row, sms=sms) == SMALL
    assert path_of(per_sm * sms + 1, K, row, sms=sms) == STREAM


@pytest.mark.parametrize("sms", [152, 76])
@pytest.mark.parametrize("resident", [False, True])
def test_clusters_up_to_a_cta_per_sm(path_of, sms, resident):
    """And with resident inputs no more clusters of eight than are resident at once."""
    for ctas, row in ((2, 20 * KB), (4, 33 * KB), (8, 65 * KB)):
        most = (14 * sms // 152) if resident and ctas == 8 else sms // ctas
        assert path_of(most, 3, row, resident=resident, sms=sms) == SMALL
        assert path_of(most + 1, 3, row, resident=resident, sms=sms) != SMALL


def test_clusters_of_four_and_eight_up_to_five_megabytes(path_of):
    assert path_of(76, 3, 30 * KB) == SMALL                       # clusters of two: 9 MB
    assert path_of(20, 3, 62 * KB) == SMALL                       # of four
    assert path_of(21, 3, 62 * KB) == STREAM
    assert path_of(10, 3, 127 * KB - 16) == SMALL                 # of eight
    assert path_of(11, 3, 127 * KB - 16) == STREAM


@pytest.mark.parametrize("sms", [152, 76])
def test_resident_rows_go_to_the_tma_pipeline_once_their_units_fill_the_gpu(path_of, sms):
    """The line between 20.6 and 23.8 MB for 152 SMs moves with the SM count, and so do three rows a slice."""
    row, B = 128 * KB, lambda mb: int(mb * 1e6 * sms / 152 / (9 * 128 * KB))
    assert path_of(B(20.6), 8, row, resident=True, sms=sms) == STREAM
    assert path_of(B(23.8), 8, row, resident=True, sms=sms) == TMA
    assert path_of(B(23.8), 8, row, resident=False, sms=sms) == STREAM
    rows = 3 * sms
    assert path_of(rows // 3, 2, 96 * KB, resident=True, single=False, sms=sms) == TMA
    assert path_of(rows // 3 + 1, 2, 96 * KB, resident=True, single=False, sms=sms) == STREAM
    assert path_of(rows // 3 + 1, 2, 112 * KB, resident=True, single=False, sms=sms) == TMA


def test_no_small_kernel_for_blocks_and_shards(path_of):
    assert path_of(1, 8, KB) == SMALL
    assert path_of(1, 8, KB, single=False) == STREAM
    assert path_of(1, 0, 508 * KB) == SMALL
    assert path_of(1, 0, 508 * KB + 16) == STREAM


def test_few_long_rows_go_to_the_tma_pipeline_from_a_megabyte_on(path_of):
    assert path_of(2, 31, 64 * KB, resident=True) == TMA          # 64 rows
    assert path_of(1, 1, 512 * KB, resident=True) == TMA          # 1 MB
    assert path_of(1, 0, MB - 16, resident=True) == STREAM
    assert path_of(13, 4, 64 * KB, resident=True, single=False) == STREAM  # 65 rows, 4 MB


def test_selection_inside_the_row_stage(path_of):
    """Large calls in long rows take the pipeline, whose CTAs count slices; without it they do not."""
    row = 192 * KB
    B = 80_000_000 // (9 * row)
    assert path_of(B + 1, 8, row, fused=True) == TMA
    assert path_of(B, 8, row, fused=True) == STREAM
    assert path_of(B + 1, 8, row - 16, fused=True) == STREAM
    assert path_of(B + 1, 8, row) == STREAM
    assert path_of(1, 8, KB, fused=True) == SMALL
