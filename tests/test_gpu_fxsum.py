"""The FP64 update where its flux differences leave the exact range of the
fixed-point sum (fv_fxsum.cuh) and take the FP64 adds instead: momenta many
orders below the pressure, zero momenta, huge and tiny scales, in one batch
with ordinary cells; against the oracle (1e-12, the FP64 tolerance), and every
patch bitwise equal to the same patch updated alone in the batch's other
layouts (CTA sizes)."""
import numpy as np
import pytest

import oracle
from paper_2302_09005_gb300 import inputs
from tests import fvtest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("d,p", [(2, 3), (2, 8), (3, 3), (3, 5), (3, 6), (3, 8)])
@pytest.mark.parametrize("uscale", [0.0, 1e-15, 1e-9, 1e-4])
def test_update_with_spread_fluxes(d, p, uscale):
    fvtest.ensure_built()
    torch = fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv
    n, s = 37, d + 2
    q, off, sz = fvtest.random_batch(n, p, d, 5)
    rng = np.random.default_rng(6)
    scale = 10.0 ** rng.integers(-100, 100, n)
    for i in range(n):
        c = q[off[i]:off[i] + (p + 2) ** d * s].reshape(-1, s)
        rho, u = c[:, 0].copy(), c[:, 1:1 + d] / c[:, :1]
        pr = rng.uniform(0.5, 1.5, len(c))
        u[:, (i % d):] *= uscale  # some directions at rest or nearly so
        c[:] = inputs.conserved_from_primitive(rho, u, pr)
        if i % 3 == 1:
            c *= scale[i]  # the whole state: densities, momenta, energies
    dx, dt = 0.01, 0.0005
    outs = []
    for nt in (32, 128, 256):
        b = fv.Batch(d, max_patch_size=p)
        tsz = fvtest.to_dev(sz)
        fv.fv_batch_plan(b.h, tsz, n)
        fv.fv_batch_set_schedule(b.h, fv.FV_SCHED_CLASSES)
        fv.fv_batch_set_class_threads(b.h, p, nt)
        x = fvtest.to_dev(q)
        y = x.clone()
        b.update(x, y, fvtest.to_dev(off), tsz, dx, dt)
        assert b.status() == fv.FV_OK
        outs.append(y.cpu().numpy())
        b.close()
    assert np.array_equal(outs[0], outs[1]) and np.array_equal(outs[0], outs[2])
    ref, _ = oracle.patch_update(q, off, sz, d, dx, dt, want_lambda=True)
    for i in range(n):  # per patch: each has its own scale
        sl = slice(off[i], off[i] + (p + 2) ** d * s)
        g, r = outs[0][sl].reshape(-1, s), ref[sl].reshape(-1, s)
        err = np.max(np.abs(g - r), axis=0)
        size = np.max(np.abs(r), axis=0)
        # a component at rest is compared at the scale of the momentum flux (p)
        size[1:1 + d] = np.maximum(size[1:1 + d], np.max(np.abs(r)))
        assert np.all(err <= 1e-12 * size), (i, err / size)
