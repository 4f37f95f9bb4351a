"""The growth of fv_run_steps' primitive buffers (csrc/fv_carry.h), compiled for
the host with an allocator of bounded memory: the library's own form where it
fits, else the documented one, nothing kept on failure, no growth where the
buffers suffice."""
import ctypes
import subprocess

import pytest

from paper_2302_09005_gb300 import _build

SRC = """
#include "fv_carry.h"
#include <map>
#include <stdlib.h>
static fv::CarryBuffers b;
static std::map<void*, int64_t> live;
static int64_t used, calls, error_at = -1;
extern "C" void reset() {
  for (auto& x : live) free(x.first);
  live.clear(); used = 0; calls = 0; error_at = -1; b = fv::CarryBuffers();
}
extern "C" void fail_at(int64_t call) { error_at = calls + call; }
// 0 ok, 1 no memory, 2 error, 3 no growth needed
extern "C" int run(int64_t full, int64_t doc, int64_t memory) {
  if (!fv::carry_must_grow(b, full, doc)) return 3;
  return (int)fv::carry_grow(b, full, doc, [&](void** p, int64_t n) {
    if (calls++ == error_at) return fv::CarryAlloc::Error;
    if (used + n > memory) return fv::CarryAlloc::NoMemory;
    *p = malloc(1); live[*p] = n; used += n;
    return fv::CarryAlloc::Ok;
  }, [&](void* p) { used -= live.at(p); live.erase(p); free(p); });
}
extern "C" int64_t state(int k) {
  return k == 0 ? b.cap : k == 1 ? b.doc : k == 2 ? used : k == 3 ? (int64_t)live.size()
       : (b.p[0] != nullptr) + (b.p[1] != nullptr);
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("carry")
    (d / "t.cpp").write_text(SRC)
    so = str(d / "t.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-I", _build.CSRC,
                    str(d / "t.cpp"), "-o", so], check=True)
    lb = ctypes.CDLL(so)
    lb.run.argtypes = [ctypes.c_int64] * 3
    lb.state.restype = ctypes.c_int64
    lb.fail_at.argtypes = [ctypes.c_int64]
    return lb


def state(lib):
    return tuple(lib.state(k) for k in range(5))


OK, NO_MEMORY, ERROR, ENOUGH = 0, 1, 2, 3


def test_own_form_where_it_fits(lib):
    lib.reset()
    assert lib.run(400, 300, 800) == OK
    assert state(lib) == (400, 0, 800, 2, 2)
    assert lib.run(400, 300, 800) == ENOUGH and lib.run(4, 3, 800) == ENOUGH


@pytest.mark.parametrize("memory", [600, 700, 799])  # the own form's second, or first, buffer
def test_documented_form_where_it_does_not(lib, memory):
    lib.reset()
    assert lib.run(400, 300, memory) == OK
    assert state(lib) == (300, 1, 600, 2, 2)
    assert lib.run(400, 300, memory) == ENOUGH  # not tried again
    assert lib.run(300, 225, memory) == ENOUGH  # the own form of a smaller run fits them
    assert lib.run(404, 303, memory) == (OK if memory >= 606 else NO_MEMORY)


def test_growth_after_the_documented_form(lib):
    lib.reset()
    assert lib.run(400, 300, 700) == OK
    assert lib.run(800, 600, 1600) == OK  # memory has become free
    assert state(lib) == (800, 0, 1600, 2, 2)


@pytest.mark.parametrize("memory", [0, 300, 599])
def test_nothing_is_kept_where_neither_fits(lib, memory):
    lib.reset()
    assert lib.run(400, 300, memory) == NO_MEMORY
    assert state(lib) == (0, 0, 0, 0, 0)
    assert lib.run(40, 30, memory) == (OK if memory >= 60 else NO_MEMORY)


@pytest.mark.parametrize("call", [0, 1])
def test_other_errors_end_the_attempt(lib, call):
    lib.reset()
    lib.fail_at(call)
    assert lib.run(400, 300, 10000) == ERROR
    assert state(lib) == (0, 0, 0, 0, 0)


def test_equal_forms(lib):  # 1D and 2D
    lib.reset()
    assert lib.run(300, 300, 600) == OK and state(lib) == (300, 0, 600, 2, 2)
    assert lib.run(301, 301, 600) == NO_MEMORY and state(lib) == (0, 0, 0, 0, 0)
