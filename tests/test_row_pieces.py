"""Pieces of rows next to the largest arc index, on the CPU: the header that
the kernels cut rows with, compiled by the host compiler, against integers
that do not wrap."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2205_14503_gb300", "csrc")
TOP = 2**32 - 2                      # the largest arc count

SHIM = """
#include "rows.h"
extern "C" void piece(uint32_t s, uint32_t e, uint32_t at, uint32_t len, uint32_t *out) {
    const stn::RowPiece p = stn::row_piece(s, e, at, len);
    out[0] = p.first;
    out[1] = p.count;
}
extern "C" uint32_t end_of(uint32_t s, uint32_t end, uint32_t len) { return stn::piece_end(s, end, len); }
extern "C" void skip(uint32_t s, uint32_t n, uint32_t step, uint32_t *out) {
    stn::RowPiece p{s, n};
    stn::skip_arcs(p, step);
    out[0] = p.first;
    out[1] = p.count;
}
"""


@pytest.fixture(scope="module")
def rows(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    src, lib = str(d / "shim.cpp"), str(d / "shim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", CSRC, src, "-o", lib], check=True)
    so = ctypes.CDLL(lib)
    so.piece.argtypes = [ctypes.c_uint32] * 4 + [ctypes.c_void_p]
    so.skip.argtypes = [ctypes.c_uint32] * 3 + [ctypes.c_void_p]
    so.end_of.argtypes = [ctypes.c_uint32] * 3
    so.end_of.restype = ctypes.c_uint32
    out = np.zeros(2, np.uint32)

    def pair(fn):
        def call(*args):
            fn(*args, out.ctypes.data)
            return int(out[0]), int(out[1])
        return call
    return pair(so.piece), pair(so.skip), so.end_of


@pytest.mark.parametrize("end", [700, 2**31 + 5, TOP - 600, TOP - 384, TOP - 31, TOP])
@pytest.mark.parametrize("degree", [0, 1, 31, 33, 127, 128, 129, 256, 511, 512, 513, 640])
def test_pieces_cover_a_row_once(rows, end, degree):
    """Chunks of 512 arcs, whole and in quarters, the one that starts past the
    row's end (the light part of a row may end chunks before the row), and
    their arcs in steps of a warp."""
    piece, skip, piece_end = rows
    start = end - degree
    for length in (128, 512):
        at, seen = 0, []
        while at < degree + 2 * 512:
            first, count = piece(start, end, at, length)
            assert count == max(0, min(degree - at, length))
            if at < degree:
                assert first == start + at and piece_end(start + at, end, length) == first + count
                for light in (start, start + at // 2, start + at, end):      # a part that ends earlier
                    assert piece_end(start + at, light, length) == max(start + at, min(light, first + count))
            while count:
                seen += range(first, first + min(32, count))
                first, count = skip(first, count, 32)
            at += length
        assert seen == list(range(start, end))
