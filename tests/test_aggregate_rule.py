"""Which lists' tile offsets are scattered and which are searched
(csrc/agg_rule.h, compiled for the host)."""
import ctypes
import subprocess

import pytest

from paper_2108_00951_gb300 import build

SOURCE = r"""
#include "agg_rule.h"
// every list's count -> bit per list: scattered
extern "C" void scattered(uint32_t n, const uint32_t* counts, uint32_t per, unsigned char* out) {
  uint32_t all = 0;
  for (uint32_t i = 0; i < n; ++i) all += efs::scatter_share(counts[i]);
  for (uint32_t i = 0; i < n; ++i) out[i] = efs::scatter_offsets(counts[i], all, per);
}
"""


@pytest.fixture(scope="module")
def scattered(tmp_path_factory):
    path = tmp_path_factory.mktemp("rule")
    (path / "r.cpp").write_text(SOURCE)
    so = str(path / "r.so")
    subprocess.run(["g++", "-O1", "-std=c++17", "-shared", "-fPIC", "-I", build.CSRC,
                    str(path / "r.cpp"), "-o", so], check=True)
    fn = ctypes.CDLL(so).scattered

    def call(counts, tiles):
        out = (ctypes.c_ubyte * len(counts))()
        fn(len(counts), (ctypes.c_uint32 * len(counts))(*counts), tiles + 1, out)
        return [bool(x) for x in out]

    return call


def test_one_list_can_hold_too_many(scattered):
    assert scattered([8 << 20], 33_779) == [True]
    assert scattered([(8 << 20) + 1], 33_779) == [False]
    assert scattered([34_600_000], 33_779) == [False]
    assert scattered([2**32 - 1], 2**20) == [False]


def test_many_long_lists_do_not_wrap_the_sum(scattered):
    assert not any(scattered([2**32 - 1] * 256, 33_779))
    assert not any(scattered([16 << 20] * 255 + [300_000], 4_000))


def test_many_lists_of_few_entries_a_tile_are_scattered(scattered):
    # 9 M entries together, but 2.2 M searches: 64 lists of 0.1 % of 138.4 M
    assert all(scattered([140_000] * 64, 33_779))
    assert all(scattered([8 * 33_780] * 256, 33_779))
    # each list by its own length
    assert scattered([64 * 33_780 - 1, 64 * 33_780] + [7 << 20], 33_779) == [True, False, False]


def test_sparse_lists_are_searched(scattered):
    assert scattered([33_780 // 16 - 1, 33_780 // 16], 33_779) == [False, True]
