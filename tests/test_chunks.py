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
extern "C" int64_t bytes_of(int64_t b, int pinned) { return fv::chunk_bytes(b, pinned != 0); }
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
    lb.bytes_of.argtypes = [ctypes.c_int64, ctypes.c_int]
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
    assert [lib.bytes_of(b, 1) for b in (0, mb, 32 * mb, 80 * mb, 2048 * mb, 1 << 40)] == \
        [4 * mb, 4 * mb, 4 * mb, 10 * mb, 256 * mb, 256 * mb]
    assert [lib.bytes_of(b, 0) for b in (0, 80 * mb, 1 << 40)] == [256 * mb] * 3
