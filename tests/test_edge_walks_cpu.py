"""The kernels' walks over edge positions, compiled for the host: near the largest edge count every thread
stays inside its edges and together they take each edge once."""
import ctypes as C
import os
import re
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1904_02241_gb300", "csrc")
LAST = 2 ** 31 - 2   # the largest edge count that a graph may have

SOURCE = r"""
#include "tc_walk.cuh"
// hits[i - first] counts position i; returns how many positions lay outside [first, end)
extern "C" long batched(uint32_t first, uint32_t end, int threads, int32_t *hits) {
    long off = 0;
    auto one = [&](uint32_t i) {
        if (i < first || i >= end) ++off; else ++hits[i - first];
    };
    for (int t = 0; t < threads && off == 0; ++t)
        tc::walk_batched<4, 1024>(first + (uint32_t)t, end, [&](uint32_t i) { for (int k = 0; k < 4; ++k) one(i + k * 1024u); }, one);
    return off;
}
// a warp's windows of 32 positions: a lane writes where it is below the end
extern "C" long windows(uint32_t first, uint32_t end, int32_t *hits) {
    long off = 0, n = 0;
    tc::walk<32>(first, end, [&](uint32_t at) {
        if (at < first || ++n > 1000) { ++off; return; }
        for (uint32_t lane = 0; lane < 32; ++lane) if (lane < end - at) ++hits[at + lane - first];
    });
    return off;
}
// a CTA's pieces of one block, with signed positions: the first `span` of a thread as loaded ahead, then the
// others one by one
extern "C" long pieces(uint32_t first, uint32_t end, int span, int32_t *hits) {
    long off = 0, n = 0;
    const int32_t r0 = (int32_t)first, r1 = (int32_t)end;
    for (int32_t t = 0; t < 512 && off == 0; ++t) {
        auto one = [&](int32_t r) {
            if (r < r0 || r >= r1 || ++n > 100000) ++off; else ++hits[r - r0];
        };
        for (int h = 0; h < span; ++h)
            if (r0 + t + h * 512 < r1) one(r0 + t + h * 512);
        for (int32_t r = r0 + t + span * 512; r < r1 && off == 0; r += 512) one(r);
    }
    return off;
}
// eight lanes along one row, as far as 64-bit positions go on from each lane's first
extern "C" long lanes(uint32_t first, uint32_t end, int32_t *hits) {
    for (int lane = 0; lane < 8; ++lane) {
        const int32_t at = tc::lane_first((int32_t)first, (int32_t)end, lane);
        for (int64_t i = at; i < (int64_t)end; i += 8) {
            if (i < (int64_t)first) return 1;
            ++hits[i - first];
        }
    }
    return 0;
}
extern "C" int most_pieces(int past) {
    int32_t n = INT32_MAX;
    while (!tc::fits_signed(n, past)) --n;
    return n;
}
"""


@pytest.fixture(scope="module")
def walks(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    d = tmp_path_factory.mktemp("walks")
    (d / "w.cpp").write_text(SOURCE)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fwrapv", "-shared", "-fPIC", "-I", CSRC, str(d / "w.cpp"), "-o", str(d / "w.so")],
                   check=True)
    return C.CDLL(str(d / "w.so"))


def _all_taken_once(f, first, end, *args):
    f.restype = C.c_long
    hits = np.zeros(max(end - first, 1), np.int32)
    off = f(C.c_uint32(first), C.c_uint32(end), *args, hits.ctypes.data_as(C.c_void_p))
    assert off == 0 and np.all(hits[:end - first] == 1)


@pytest.mark.parametrize("end", [LAST, LAST - 1, LAST - 1023, LAST - 4096, 5000, 4096, 1])
@pytest.mark.parametrize("n", [0, 1, 1023, 1024, 1025, 3072, 3073, 4097, 9000])
def test_push_tiles_stay_inside_their_edges(walks, end, n):
    _all_taken_once(walks.batched, max(end - n, 0), end, C.c_int(1024))


@pytest.mark.parametrize("end", [LAST, LAST - 1, LAST - 31, LAST - 32, 2048, 1])
@pytest.mark.parametrize("n", [0, 1, 31, 32, 33, 40, 2048])
def test_row_ids_of_the_last_edges(walks, end, n):
    _all_taken_once(walks.windows, max(end - n, 0), end)


def _constant(file, name):
    text = open(os.path.join(CSRC, file)).read()
    m = re.search(r"constexpr int " + name + r" = ([0-9]+)(?: \* SPM_THREADS)?;", text)
    return int(m.group(1))


@pytest.mark.parametrize("n", [0, 1, 511, 512, 513, 2049, 5000])
@pytest.mark.parametrize("span", [1, 2, 4])
def test_last_pieces_of_the_largest_staged_product(walks, n, span):
    """Up to as many pieces as the staged product takes, its signed positions do not wrap."""
    threads = _constant("tc_spmv.cu", "SPM_THREADS")
    assert threads == 512
    end = walks.most_pieces(C.c_int(_constant("tc_spmv.cu", "SPM_PAST") * threads))
    assert end < LAST - span * threads
    _all_taken_once(walks.pieces, end - n, end, C.c_int(span))


@pytest.mark.parametrize("end", [LAST, LAST - 6, LAST - 7, 64])
@pytest.mark.parametrize("n", [0, 1, 7, 8, 9, 64])
def test_lanes_of_the_last_rows(walks, end, n):
    _all_taken_once(walks.lanes, end - n, end)
