"""How the host pipeline cuts a batch into chunks (csrc/fv_chunks.h), compiled
for the host: by bytes, whatever patch comes first.  Every chunk spans at most
its byte target unless it is one patch, could not take the next patch as
well, and the chunks cover the batch in order."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_2302_09005_gb300 import _build

SRC = """
#include "fv_chunks.h"
extern "C" int64_t bytes_of(int64_t b, int64_t box, int pinned) {
  return fv::chunk_bytes(b, box, pinned != 0);
}
extern "C" int64_t end_of(int64_t p0, int64_t n, const int64_t* off, const int64_t* len, int64_t es,
                          int64_t want) {
  return fv::chunk_end(p0, n, off, [&](int64_t i) { return len[i]; }, es, want);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("chunks")
    (d / "t.cpp").write_text(SRC)
    so = str(d / "t.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", _build.CSRC,
                    str(d / "t.cpp"), "-o", so], check=True)
    lb = ctypes.CDLL(so)
    lb.bytes_of.restype = lb.end_of.restype = ctypes.c_int64
    lb.bytes_of.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_int]
    lb.end_of.argtypes = [ctypes.c_int64, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p,
                          ctypes.c_int64, ctypes.c_int64]
    return lb


def cut(lib, off, ln, es, want):
    n, p0, out = len(off), 0, [0]
    while p0 < n:
        p0 = lib.end_of(p0, n, off.ctypes.data, ln.ctypes.data, es, want)
        out.append(p0)
    return out


KINDS = {"uniform": lambda r: np.full(900, 8), "one": lambda r: np.array([8]),
         "small_first": lambda r: np.r_[1, np.full(899, 8)],
         "large_first": lambda r: np.r_[8, np.full(5000, 1)],
         "ragged": lambda r: r.integers(1, 9, 2000),
         "ascending": lambda r: np.sort(r.integers(1, 9, 2000))}


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("gap", [0, 2000, "random"])
@pytest.mark.parametrize("want", [1, 40000, 1 << 20, 4 << 20, 1 << 40])
def test_chunks_by_bytes(lib, kind, gap, want):
    rng = np.random.default_rng(6)
    p = KINDS[kind](rng).astype(np.int64)
    es, ln = 8, (p + 2) ** 3 * 5
    pitch = ln + (rng.integers(0, 20000, len(p)) if gap == "random" else gap)
    off = np.r_[0, np.cumsum(pitch)[:-1]].astype(np.int64) + 16
    c = cut(lib, off, ln, es, want)
    assert c[0] == 0 and c[-1] == len(p) and all(a < b for a, b in zip(c, c[1:]))
    for a, b in zip(c, c[1:]):
        assert b == a + 1 or (off[b - 1] + ln[b - 1] - off[a]) * es <= want
        assert b == len(p) or (off[b] + ln[b] - off[a]) * es > want


def test_chunk_bytes_bounds(lib):
    mb = 1 << 20
    sizes = (0, mb, 32 * mb, 80 * mb, 2048 * mb, 1 << 40)
    assert [lib.bytes_of(b, 1, 1) for b in sizes] == \
        [4 * mb, 4 * mb, 4 * mb, 10 * mb, 256 * mb, 256 * mb]
    assert lib.bytes_of(80 * mb, 5, 1) == 10 * mb + 4
    assert [lib.bytes_of(b, 5, 0) for b in sizes] == [256 * mb] * 6


@pytest.mark.parametrize("kind", sorted(KINDS))
@pytest.mark.parametrize("copies", [3, 7, 8, 9])
def test_eight_chunks_hold_the_batch(lib, kind, copies):
    """From 32 MB to 2 GB; patches a little further apart than they are long."""
    rng = np.random.default_rng(copies)
    p = np.tile(KINDS[kind](rng), copies * (1000 if kind == "one" else 3)).astype(np.int64)
    ln = (p + 2) ** 3 * 5
    off = np.r_[0, np.cumsum(ln + 1)[:-1]].astype(np.int64)
    total = int(off[-1] + ln[-1]) * 8
    want = lib.bytes_of(total, 10 ** 3 * 5 * 8, 1)
    c = cut(lib, off, ln, 8, want)
    assert total < 2 << 30 and (want == 4 << 20 or len(c) - 1 <= 8)
    if kind == "uniform":
        assert c[1] == -(-len(p) // 8)
