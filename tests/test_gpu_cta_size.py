"""Launches without a plan choose the CTA size themselves (by precision, patch
size and batch size); a planned launch with a set size must give the same bits,
at the sizes on both sides of each line."""
import numpy as np
import pytest

from paper_2302_09005_gb300 import inputs
from tests import fvtest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,p", [(2, 7), (2, 8), (2, 9), (2, 12), (2, 13), (2, 19), (2, 20), (2, 24),
                                 (3, 3), (3, 4), (3, 5), (3, 6), (3, 7), (3, 8)])
@pytest.mark.parametrize("n", [7, 1300])
@pytest.mark.parametrize("prec", [0, 1])
def test_untuned_launch_equals_set_cta_size(d, p, n, prec):
    fvtest.ensure_built()
    torch = fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv
    q, off, sz = fvtest.random_batch(n, p, d, 11, dtype=np.float32 if prec else np.float64)
    nbr = fvtest.to_dev(inputs.self_periodic_neighbours(n, d))
    toff, tsz = fvtest.to_dev(off), fvtest.to_dev(sz)
    dx, cfl = 0.01, 0.4
    mask = fvtest.interior_mask(off, sz, d, d + 2, len(q))
    got = []
    for nt in (None, 128):
        b = fv.Batch(d, precision=prec, max_patch_size=p)
        if nt is not None:
            fv.fv_batch_plan(b.h, tsz, n)
            fv.fv_batch_set_schedule(b.h, fv.FV_SCHED_CLASSES)
            fv.fv_batch_set_class_threads(b.h, p, nt)
        x, y = fvtest.to_dev(q), fvtest.to_dev(q)
        u = x.clone()
        lam = torch.zeros(n, dtype=torch.float64, device="cuda")
        b.update(x, u, toff, tsz, dx, 0.001, lambda_patch=lam)
        pa = torch.empty(n * b.prim_stride(), dtype=x.dtype, device="cuda")
        b.halo_fill(x, toff, tsz, nbr)
        b.max_eigenvalue(x, toff, tsz, cfl, dx)
        b.time_step_prim(x, y, None, pa, toff, tsz, nbr, dx, cfl)
        assert b.status() == fv.FV_OK
        got.append((u.cpu().numpy()[mask], lam.cpu().numpy(), y.cpu().numpy()[mask],
                    fv.fv_read_dt(b.h)))
        b.close()
    assert all(np.array_equal(a, c) for a, c in zip(*got))
