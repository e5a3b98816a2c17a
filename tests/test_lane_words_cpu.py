"""The addresses of the unpacking kernels at width 3 on the host (csrc/skim_lane_words.h): no lane reads a word behind the row's last one, and the
words it reads hold the codes it owns."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "skim_lane_words.h"
#include <stdint.h>
// As the kernel goes through a row: whole steps of 256 columns, then the lanes of the last one that have columns.
// Returns the highest word read; codes: [cols]
extern "C" int unpack_row(const uint32_t *row, int cols, uint8_t *codes)
{
    int highest = -1;
    for (int t = 0; t * 256 < cols; ++t)
        for (int lane = 0; lane < 32; ++lane) {
            const int j = t * 256 + lane * 8;
            if (j >= cols) continue;
            const int columns = (t + 1) * 256 <= cols ? 8 : cols - j;
            const SkimLaneWords3 w(lane);
            const int first = t * 24 + w.first, last = first + (w.reaches_next(columns) ? 1 : 0);
            highest = last > highest ? last : highest;
            const uint64_t both = row[first] | (last > first ? (uint64_t)row[last] << 32 : 0);
            for (int u = 0; u < 8 && j + u < cols; ++u) codes[j + u] = (uint8_t)(both >> (w.shift + 3 * u) & 7);
        }
    return highest;
}
"""


@pytest.fixture(scope="module")
def unpack(tmp_path_factory):
    d = tmp_path_factory.mktemp("lane_words")
    src, lib = d / "lane_words.cpp", d / "lane_words.so"
    src.write_text(SOURCE)
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I", os.path.join(ROOT, "paper_2412_04180_b200", "csrc"), "-o", str(lib), str(src)],
                   check=True)
    f = ctypes.CDLL(str(lib)).unpack_row
    f.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_void_p]
    f.restype = ctypes.c_int
    return f


def test_lanes_stay_inside_their_row(unpack):
    """Every row length to three steps: 41, 42, 81 .. 85 modulo 128 are those whose last codes end in the last of the row's four words while a
    whole group of eight would reach into the next."""
    rng = np.random.default_rng(5)
    for cols in range(1, 769):
        want = rng.integers(0, 8, cols).astype(np.uint8)
        words = (cols * 3 + 31) // 32
        bits = np.unpackbits(want[:, None], axis=1, bitorder="little")[:, :3].reshape(-1)
        row = np.packbits(np.pad(bits, (0, words * 32 - bits.size)), bitorder="little").view("<u4").copy()
        got = np.zeros(cols, np.uint8)
        assert unpack(np.pad(row, (0, 1)).ctypes.data, cols, got.ctypes.data) < words, cols      # (the last word written, which padding may follow)
        np.testing.assert_array_equal(got, want)
