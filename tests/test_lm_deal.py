"""The fused LM head's cut into items and their deal to the CTA pairs, compiled with the host compiler."""
import ctypes
import subprocess

import pytest

from paper_2608_03447_gb300 import build

SHIM = """
#include "asd_lm_deal.h"
extern "C" void deal(int T, int V, int kw, int pairs, int* out) {
  const asd_detail::LmDeal d = asd_detail::lm_deal(T, V, kw, pairs);
  out[0] = d.tn;
  out[1] = d.token_tiles;
  out[2] = d.full;
  out[3] = d.entries;
}
extern "C" int rows_per_launch(int V) { return asd_detail::lm_rows_per_launch(V); }
extern "C" int logits_in_two_tiles(int V, int pairs) { return asd_detail::lm_logits_in_two_tiles(V, pairs); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("deal")
    (d / "shim.cpp").write_text(SHIM)
    out = str(d / "shim.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-Wall", "-Werror", "-shared", "-fPIC", f"-I{build.CSRC}",
                    str(d / "shim.cpp"), "-o", out], check=True)
    return ctypes.CDLL(out)


def _deal(lib, T, V, kw, pairs=76):
    out = (ctypes.c_int * 4)()
    lib.deal(T, V, kw, pairs, out)
    return tuple(out)


BIG = 2**31 - 1


@pytest.mark.parametrize("V", [1, 256, 257, 512, 513, 9717, 38912, 39424, 151936, 1 << 24, 1 << 30, BIG])
@pytest.mark.parametrize("T", [1, 32, 33, 256, 257, 600, 2304, 65536, 1 << 17, 1 << 24, BIG])
def test_items_of_a_launch_fit_32_bits(lib, T, V):
    """Every tile of token rows by every unit of vocabulary rows is an item, also at the largest sizes; a launch
    of the most rows leaves room for the pairs' stride behind the last entry."""
    most = lib.rows_per_launch(V)
    assert most >= 65536 and most % 256 == 0
    T = min(T, most)
    for kw in (1, 2) if T <= 256 else (2,):
        tn, tiles, full, entries = _deal(lib, T, V, kw)
        assert tn % 32 == 0 and 32 <= tn <= 256 and tiles * tn >= T
        items = -(-V // (256 * kw)) * tiles
        assert full <= items <= entries <= 2**31 - 1 - 76
        assert full + (entries - full) // (1 if entries == items else 2) == items
        assert (entries - full) % 2 == 0 or entries == full


@pytest.mark.parametrize("T,V,tiles,tn", [
    (477, 12800, 3, 160), (477, 12801, 2, 256),     # 75 items of three tiles are one round, 78 are not
    (477, 9728, 2, 256), (477, 9729, 3, 160),       # 38 items go in halves, 40 do not
    (600, 9717, 4, 160), (600, 9729, 3, 224),       # 76 and 80 items
    (300, 12509, 2, 160), (384, 12509, 2, 192), (385, 12509, 3, 160),
    (2304, 151936, 9, 256), (576, 151936, 3, 192)])
def test_one_round_of_narrower_tiles(lib, T, V, tiles, tn):
    assert _deal(lib, T, V, 2)[:2] == (tn, tiles)


def test_logits_of_one_tile(lib):
    assert [lib.logits_in_two_tiles(V, 76) for V in (19456, 19457, 24320, 24321, 151936)] == [0, 1, 1, 0, 0]
