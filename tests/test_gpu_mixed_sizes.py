"""Launches that mix patch sizes, where every size runs in its own or in the
runtime-size code of one kernel and small patches share a large patch's CTA:
the same bits as one launch per size with 128 threads, for updates, time steps
and the handed-on primitives."""
import numpy as np
import pytest

from paper_2302_09005_gb300 import inputs
from tests import fvtest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,pmax", [(2, 4), (2, 8), (2, 11), (2, 17), (2, 19), (2, 22), (2, 24),
                                    (3, 3), (3, 4), (3, 5), (3, 6), (3, 7), (3, 8), (3, 9)])
@pytest.mark.parametrize("prec", [0, 1])
def test_mixed_launch_equals_class_launches(d, pmax, prec):
    fvtest.ensure_built()
    torch = fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv
    dtype = np.float32 if prec else np.float64
    n = 700
    sizes = np.random.default_rng(pmax).integers(1, pmax + 1, n).astype(np.int32)
    q, off, sz = inputs.random_batch(n, sizes, d, seed=12, dtype=dtype)
    nbr = fvtest.to_dev(inputs.self_periodic_neighbours(n, d))
    toff, tsz = fvtest.to_dev(off), fvtest.to_dev(sz)
    dx, cfl = 0.01, 0.4
    mask = fvtest.interior_mask(off, sz, d, d + 2, len(q))
    got = []
    for planned in (False, True):
        b = fv.Batch(d, precision=prec, max_patch_size=pmax)
        if planned:
            fv.fv_batch_plan(b.h, tsz, n)
            fv.fv_batch_set_schedule(b.h, fv.FV_SCHED_CLASSES)
            for p in range(1, pmax + 1):
                fv.fv_batch_set_class_threads(b.h, p, 128)
        x, y = fvtest.to_dev(q), fvtest.to_dev(q)
        u, w = x.clone(), x.clone()
        lam = torch.zeros(n, dtype=torch.float64, device="cuda")
        b.update(x, u, toff, tsz, dx, 0.001, lambda_patch=lam)
        pa = torch.zeros(n * b.prim_stride(), dtype=x.dtype, device="cuda")
        pb = torch.zeros_like(pa)
        b.halo_fill(x, toff, tsz, nbr)
        b.max_eigenvalue(x, toff, tsz, cfl, dx)
        b.time_step(x, w, toff, tsz, nbr, dx, cfl)
        dt = fv.fv_read_dt(b.h)
        b.max_eigenvalue(x, toff, tsz, cfl, dx)
        b.time_step_prim(x, y, None, pa, toff, tsz, nbr, dx, cfl)
        b.time_step_prim(y, x, pa, pb, toff, tsz, nbr, dx, cfl)
        r0, r1 = fvtest.to_dev(q), fvtest.to_dev(q)
        b.run_steps(r0, r1, toff, tsz, nbr, dx, cfl, 3)
        assert b.status() == fv.FV_OK
        got.append([u.cpu().numpy()[mask], lam.cpu().numpy(), w.cpu().numpy()[mask], np.array(dt),
                    pa.cpu().numpy(), pb.cpu().numpy(), x.cpu().numpy()[mask],
                    r1.cpu().numpy()[mask]])
        b.close()
    for a, c in zip(*got):
        assert np.array_equal(a, c)
