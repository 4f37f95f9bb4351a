"""The largest patch size a handle accepts (one shared-memory stage of the
general kernel) and the first it refuses, and a step at the largest size on
every path that sizes its own shared memory (update, time step, carry)."""
import numpy as np
import pytest

import oracle
from tests import fvtest

pytestmark = pytest.mark.gpu

# (precision, d): the largest max_patch_size
LIMITS = {(0, 2): 40, (0, 3): 9, (1, 2): 57, (1, 3): 12}


@pytest.mark.parametrize("prec,d", sorted(LIMITS))
def test_largest_patch_size(prec, d):
    fvtest.ensure_built()
    torch = fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv, inputs
    p = LIMITS[prec, d]
    with pytest.raises(fv.FvError) as e:
        fv.Batch(d, precision=prec, max_patch_size=p + 1)
    assert e.value.status == fv.FV_ERR_UNSUPPORTED
    n, dx = 5, 0.01
    q, off, sz = fvtest.random_batch(n, p, d, 3, np.float32 if prec else np.float64)
    nbr = inputs.self_periodic_neighbours(n, d)
    toff, tsz, tnbr = (fvtest.to_dev(a) for a in (off, sz, nbr))
    b = fv.Batch(d, precision=prec, max_patch_size=p)
    x = fvtest.to_dev(q)
    y = x.clone()
    b.run_steps(x, y, toff, tsz, tnbr, dx, 0.4, 3)
    assert b.status() == fv.FV_OK
    ref = q.astype(np.float64)
    for _ in range(3):
        ref, _ = oracle.step(ref, off, sz, nbr, d, dx, 0.4)
    s = d + 2
    mask = fvtest.interior_mask(off, sz, d, s, len(q))
    err = fvtest.per_unknown_rel_err(y.cpu().numpy(), ref, mask, s)
    assert np.all(err <= (1e-5 if prec else 1e-12)), err
    b.close()
