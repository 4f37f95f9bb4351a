"""Launches that start under the ones before them (programmatic dependent
launch): a chain of calls on one stream, fed by torch kernels just before it and
read just after it, gives bitwise what the same calls give with the device
synchronised between all of them -- for one patch, for launches below and above
the size where ordinary launches overlap, for size classes, and in a captured
graph replayed several times."""
import numpy as np
import pytest

from paper_2302_09005_gb300 import inputs
from tests import fvtest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fv():
    fvtest.ensure_built()
    fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv as fvmod
    return fvmod


def chain(fv, torch, b, st, src, off, sz, nbr, n, s, classes, sync):
    """Copies of the inputs made by torch kernels, then every kind of call."""
    def wait():
        if sync:
            torch.cuda.synchronize()
    with torch.cuda.stream(st):
        x, toff, tsz, tnbr = src.clone(), off.clone(), sz.clone(), nbr.clone()
        y = torch.zeros_like(x)
        if classes:
            fv.fv_batch_plan(b.h, tsz, n)
            fv.fv_batch_set_schedule(b.h, fv.FV_SCHED_CLASSES)
        lam = torch.zeros(n, dtype=torch.float64, device="cuda")
        sums = torch.zeros((n, s), dtype=torch.float64, device="cuda")
        tot = torch.zeros(s, dtype=torch.float64, device="cuda")
        out = []
        wait()
        b.halo_fill(x, toff, tsz, tnbr)
        wait()
        b.max_eigenvalue(x, toff, tsz, 0.4, 0.01, per_patch=lam)
        wait()
        b.update(x, y, toff, tsz, 0.01, -1.0)
        wait()
        fv.fv_patch_sums(b.h, y, toff, tsz, n, sums, tot)
        wait()
        out += [y.clone(), lam.clone(), sums, tot]
        for _ in range(3):
            b.time_step(x, y, toff, tsz, tnbr, 0.01, 0.4)
            wait()
            b.time_step(y, x, toff, tsz, tnbr, 0.01, 0.4, lambda_patch=lam)
            wait()
        out += [x.clone(), lam.clone()]
        b.run_steps(x, y, toff, tsz, tnbr, 0.01, 0.4, 5)
        wait()
        out += [y.clone()]
    torch.cuda.synchronize()
    assert b.status() == fv.FV_OK
    return out


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("d,sizes,n", [(2, (3,), 1), (2, (3,), 64), (3, (5,), 303), (2, (5,), 5000),
                                       (3, (3, 5, 7), 120), (3, (2, 4, 6, 8), 700),
                                       (3, (3, 5, 7), 6000)])
def test_chain_equals_synchronised_calls(fv, prec, d, sizes, n):
    torch = fvtest.torch_cuda()
    rng = np.random.default_rng(n)
    psz = rng.choice(sizes, n).astype(np.int32)
    q, off, _ = inputs.random_batch(n, psz, d, seed=4, dtype=np.float32 if prec else np.float64)
    nbr = inputs.self_periodic_neighbours(n, d)
    src, toff, tsz, tnbr = (fvtest.to_dev(a) for a in (q, off, psz, nbr))
    st = torch.cuda.Stream()
    torch.cuda.synchronize()
    for classes in (False, True):
        b = fv.Batch(d, precision=prec, max_patch_size=max(sizes), stream=st)
        args = (fv, torch, b, st, src, toff, tsz, tnbr, n, d + 2, classes)
        ref = chain(*args, True)
        for _ in range(5):
            for r, g in zip(ref, chain(*args, False)):
                assert torch.equal(r, g)
        b.close()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("steps", [1, 2])
def test_captured_time_steps_replay(fv, prec, steps):
    """A caller's own graph of one or two time steps, replayed: every replay
    finds the wave speed where an eager step would."""
    torch = fvtest.torch_cuda()
    d, p, n = 2, 4, 30
    q, off, sz = fvtest.random_batch(n, p, d, 6, np.float32 if prec else np.float64)
    nbr = inputs.self_periodic_neighbours(n, d)
    toff, tsz, tnbr = (fvtest.to_dev(a) for a in (off, sz, nbr))
    res = []
    for graph in (False, True):
        st = torch.cuda.Stream()
        x, y = fvtest.to_dev(q), fvtest.to_dev(q)
        torch.cuda.synchronize()
        b = fv.Batch(d, precision=prec, max_patch_size=p, stream=st)
        b.halo_fill(x, toff, tsz, tnbr)
        b.max_eigenvalue(x, toff, tsz, 0.4, 0.01)

        def body():
            b.time_step(x, y, toff, tsz, tnbr, 0.01, 0.4)
            if steps == 2:
                b.time_step(y, x, toff, tsz, tnbr, 0.01, 0.4)

        torch.cuda.synchronize()
        if graph:
            g = torch.cuda.CUDAGraph()
            with torch.cuda.graph(g, stream=st):
                body()
            for _ in range(4):
                with torch.cuda.stream(st):
                    g.replay()
        elif steps == 2:
            for _ in range(4):
                body()
        else:  # a replayed single step repeats itself: same input, same wave speed
            body()
        torch.cuda.synchronize()
        res.append((x.clone(), y.clone(), fv.fv_read_dt(b.h)))
        assert b.status() == fv.FV_OK
        b.close()
    assert torch.equal(res[0][0], res[1][0]) and torch.equal(res[0][1], res[1][1])
    assert res[0][2] == res[1][2]


@pytest.mark.parametrize("prec", [0, 1])
def test_event_waits_hold(fv, prec):
    """A launch after a wait on another stream's event sees what that stream
    wrote, although the kernel before it on its own stream lets it start early:
    the other stream is kept busy, then changes the input."""
    torch = fvtest.torch_cuda()
    d, p, n = 2, 4, 20
    q, off, sz = fvtest.random_batch(n, p, d, 7, np.float32 if prec else np.float64)
    toff, tsz = fvtest.to_dev(off), fvtest.to_dev(sz)
    old, new = fvtest.to_dev(q), fvtest.to_dev(q) * 1.25
    one, two = torch.cuda.Stream(), torch.cuda.Stream()
    x, y, ref = old.clone(), torch.zeros_like(old), torch.zeros_like(old)
    torch.cuda.synchronize()
    b = fv.Batch(d, precision=prec, max_patch_size=p, stream=one)
    b.update(new, ref, toff, tsz, 0.01, 1e-3)
    torch.cuda.synchronize()
    for _ in range(5):
        x.copy_(old)
        y.zero_()
        torch.cuda.synchronize()
        ev = torch.cuda.Event()
        with torch.cuda.stream(two):
            torch.cuda._sleep(2_000_000)  # about a millisecond
            x.copy_(new)
            ev.record(two)
        b.update(old, y, toff, tsz, 0.01, 1e-3)  # its end lets the next one start
        one.wait_event(ev)
        b.update(x, y, toff, tsz, 0.01, 1e-3)
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
    assert b.status() == fv.FV_OK
    b.close()
