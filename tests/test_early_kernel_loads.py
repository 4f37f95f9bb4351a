"""Kernels that may start while the kernel before them still runs read what that
kernel writes by ordinary loads only: griddepcontrol.wait does not order the
non-coherent path (ld.global.nc: __ldg, or pointers to const that __restrict__
lets the compiler read so).  Checked in their sources: the files that launch
through launch_kernel() and every header these include.  The one exception is
the training kernel's samples, which no kernel of a training call writes."""
import os
import re

import pytest

from paper_2302_09005_gb300 import _build

SAMPLES = {"fv_mlp.cu": [r"__ldg\(reinterpret_cast<const float4\*>\(a\.[xt] \+"]}
NC = [r"__ldg\s*\(", r"ld\.global(\.\w+)*\.nc", r"const\s+\w+\s*\*\s*__restrict__\s+\w+\s*[;,)]"]


def code(name):
    s = open(os.path.join(_build.CSRC, name)).read()
    return re.sub(r"//[^\n]*|/\*.*?\*/", "", s, flags=re.S)


def early_sources():
    names = {os.path.basename(f) for f in _build.sources()}
    names |= {f for f in os.listdir(_build.CSRC) if f.endswith((".cuh", ".h"))}
    todo = [f for f in names if re.search(r"\blaunch_kernel\(", code(f))]
    seen = set()
    while todo:
        f = todo.pop()
        if f in names and f not in seen:
            seen.add(f)
            todo += re.findall(r'#include "([^"]+)"', code(f))
    return sorted(seen)


def test_the_early_kernels_are_found():
    assert {"fv_step.cuh", "fv_rows2d.cu", "fv_march3d.cu", "fv_halo.cu", "fv_reduce.cu",
            "fv_mlp.cu", "fv_meta.cuh"} <= set(early_sources())


@pytest.mark.parametrize("name", early_sources())
def test_no_non_coherent_loads(name):
    s = code(name)
    for allowed in SAMPLES.get(name, []):
        s = re.sub(allowed, "", s)
    for pat in NC:
        assert not re.search(pat, s), (name, pat)
