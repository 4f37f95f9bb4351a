"""CTA sizes that FP64 launches really take, read from a captured graph of one
call: a launch per size goes by that size, one launch by the handle's largest;
a class whose CTA size was set goes back to the launch's own choice with 0."""
import ctypes

import numpy as np
import pytest

from paper_2302_09005_gb300 import inputs
from tests import fvtest

pytestmark = pytest.mark.gpu


class KernelNode(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("grid", ctypes.c_uint * 3),
                ("block", ctypes.c_uint * 3), ("shared", ctypes.c_uint),
                ("params", ctypes.c_void_p), ("extra", ctypes.c_void_p),
                ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def kernel_threads(stream, call):
    """Threads per CTA of the kernels that call() launches on the stream."""
    cu = ctypes.CDLL("libcuda.so.1")
    vp = ctypes.c_void_p

    def ok(r):
        assert r == 0, r
    call()  # the library's own first-use work happens outside the capture
    stream.synchronize()
    s = vp(stream.cuda_stream)
    ok(cu.cuStreamBeginCapture_v2(s, 1))
    call()
    graph = vp()
    ok(cu.cuStreamEndCapture(s, ctypes.byref(graph)))
    n = ctypes.c_size_t(0)
    ok(cu.cuGraphGetNodes(graph, None, ctypes.byref(n)))
    nodes = (vp * n.value)()
    ok(cu.cuGraphGetNodes(graph, nodes, ctypes.byref(n)))
    out = []
    for node in nodes:
        kind = ctypes.c_int(-1)
        ok(cu.cuGraphNodeGetType(vp(node), ctypes.byref(kind)))
        if kind.value == 0:
            k = KernelNode()
            ok(cu.cuGraphKernelNodeGetParams_v2(vp(node), ctypes.byref(k)))
            out.append(int(k.block[0]))
    ok(cu.cuGraphDestroy(graph))
    return out


def batch(fv, d, p, n, pmax):
    torch = fvtest.torch_cuda()
    stream = torch.cuda.Stream()
    q, off, sz = inputs.random_batch(n, p, d, seed=1)
    b = fv.Batch(d, max_patch_size=pmax, stream=stream)
    x, toff, tsz = fvtest.to_dev(q), fvtest.to_dev(off), fvtest.to_dev(sz)
    y = x.clone()
    torch.cuda.synchronize()
    return b, tsz, stream, lambda: b.update(x, y, toff, tsz, 0.01, 0.001)


@pytest.fixture(scope="module")
def fv():
    fvtest.ensure_built()
    fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv as fvmod
    return fvmod


@pytest.mark.parametrize("p,pmax,threads", [(5, 12, 64), (5, 19, 128), (5, 20, 256), (12, 12, 64),
                                            (19, 19, 128), (20, 20, 256)])
@pytest.mark.parametrize("schedule", [None, 0, 2])  # no plan, one launch, a launch per size
def test_own_choice(fv, p, pmax, threads, schedule):
    b, tsz, stream, call = batch(fv, 2, p, 3000, pmax)
    if schedule is not None:
        fv.fv_batch_plan(b.h, tsz, 3000)
        fv.fv_batch_set_schedule(b.h, schedule)
    if schedule == 2 and p == 5:
        threads = 32  # the class's own size
    assert kernel_threads(stream, call) == [threads]
    b.close()


def test_zero_takes_the_launchs_own_choice(fv):
    b, tsz, stream, call = batch(fv, 3, 4, 3000, 4)
    fv.fv_batch_plan(b.h, tsz, 3000)
    fv.fv_batch_set_schedule(b.h, fv.FV_SCHED_CLASSES)
    own = kernel_threads(stream, call)
    assert own == [64]
    default = fv.fv_batch_class_threads(b.h, 4)
    fv.fv_batch_set_class_threads(b.h, 4, 128)
    assert kernel_threads(stream, call) == [128] and fv.fv_batch_class_threads(b.h, 4) == 128
    fv.fv_batch_set_class_threads(b.h, 4, 0)
    assert kernel_threads(stream, call) == own and fv.fv_batch_class_threads(b.h, 4) == default
    b.close()
