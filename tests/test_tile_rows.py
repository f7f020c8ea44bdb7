"""Rows of the interior kernel's tiles on very wide bodies: the stores of a
tile of the most rows it may have, by 32-bit byte offsets, reach the elements
they are meant for (the host code compiled on its own; no body is run)."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2208_13769_gb300", "csrc")
THREADS = 128
PAD = 3  # kPadRows
SRC = """
#include "lbm_tile_rows.h"
extern "C" int max_rows(long long pitch, int word) { return lbm::interior_max_rows(pitch, word, %d); }
extern "C" void bounded(int* rows, int* count, int h, int max) {
    lbm::ChunkLevels L;
    memcpy(L.rows, rows, sizeof(L.rows));
    memcpy(L.count, count, sizeof(L.count));
    L = lbm::bounded_chunks(L, h, max);
    memcpy(rows, L.rows, sizeof(L.rows));
    memcpy(count, L.count, sizeof(L.count));
}
""" % THREADS


@pytest.fixture(scope="module")
def host(tmp_path_factory):
    d = tmp_path_factory.mktemp("rows")
    (d / "rows.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-Wall", "-Werror", "-fPIC", "-shared", "-I", CSRC, "-o",
                    str(d / "rows.so"), str(d / "rows.cpp")], check=True)
    L = C.CDLL(str(d / "rows.so"))
    L.max_rows.argtypes = [C.c_longlong, C.c_int]
    return L


def _offsets_reach(rows, pitch, word, up):
    """The kernel's offsets over a tile's walk against the elements' places."""
    n = rows + 4
    off = ((n - 1) * pitch if up else 0) % 2 ** 32  # row a of stage A, thread 0
    step = (-pitch if up else pitch) % 2 ** 32
    for q in range(n):
        if q >= 4:  # stage C stores the row two before
            o = (off - 2 * step) % 2 ** 32
            for t in (0, THREADS - 1):
                true = ((n - 1 - q + 2 if up else q - 2) * pitch + t) * word
                if ((o + t) % 2 ** 32 * word) % 2 ** 32 != true:
                    return False
        off = (off + step) % 2 ** 32
    return True


@pytest.mark.parametrize("word", [8, 4])
@pytest.mark.parametrize("ny", [8, 12, 13, 14, 15, 20, 64, 1000])
def test_offsets_of_the_tallest_tile_fit(host, word, ny):
    """At the widest plane of so many rows that a body may have, and below."""
    widest = (2 ** 31 - 1) // (ny + 2 * PAD) // 64 * 64
    for pitch in {widest // k // 64 * 64 for k in (1, 2, 3, 4, 5, 7, 10, 30, 1000)}:
        rows = host.max_rows(pitch, word)
        assert rows >= 1
        used = min(rows, ny)
        for up in (False, True):
            assert _offsets_reach(used, pitch, word, up), (pitch, used, up)
        if rows < ny:  # the limit is not lower than it needs to be
            assert not _offsets_reach(rows + 1, pitch, word, False)


def test_a_body_of_sixty_million_by_twelve_nodes(host):
    """FP64, 253 GB: the last row of a tile of 8 would lie beyond 2^32 bytes."""
    rows = host.max_rows(59_700_000 // 64 * 64 + 64, 8)
    assert rows == 7


@pytest.mark.parametrize("rows,count,h,most", [
    ([8, 0, 0, 0], [2, 0, 0, 0], 16, 7), ([30, 10, 8, 0], [3, 2, 2, 0], 120, 9), ([30, 10, 8, 0], [3, 2, 2, 0], 120, 40),
    ([8, 4, 0, 0], [1, 1, 0, 0], 5, 6), ([18, 0, 0, 0], [1, 0, 0, 0], 3, 3)])
def test_chunks_within_the_limit_cover_the_rows(host, rows, count, h, most):
    r, n = (C.c_int * 4)(*rows), (C.c_int * 4)(*count)
    host.bounded(r, n, h, most)
    y, tallest = 0, 0
    for k in range(4):
        for _ in range(n[k]):
            if y < h:
                tallest = max(tallest, min(r[k], h - y))
                y += r[k]
    assert y >= h and tallest <= most
    if max(rows) <= most:
        assert list(r) == rows and list(n) == count
