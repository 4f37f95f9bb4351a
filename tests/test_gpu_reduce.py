"""The reductions at the edges of their work split: conservation sums for
patch sizes around the lanes and rounds of a warp and patch counts around a
cluster's chunk, against math.fsum per patch (1e-14 of the sum of magnitudes,
the totals' tolerance) and bitwise the same from run to run."""
import math

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


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("d,sizes,n", [
    (1, (1, 2, 31, 32, 33, 64, 65), 70), (2, (1, 5, 6, 8, 9, 10, 11, 12, 16, 17), 1025),
    (3, (1, 2, 3, 4, 5, 6, 7, 8), 2077), (3, (6,), 1), (2, (17,), 33), (3, (5,), 1024)])
def test_sums_at_the_edges(fv, prec, d, sizes, n):
    torch = fvtest.torch_cuda()
    s = d + 2
    rng = np.random.default_rng(n)
    sz = rng.choice(sizes, n).astype(np.int32)
    q, off, _ = inputs.random_batch(n, sz, d, seed=3, dtype=np.float32 if prec else np.float64)
    b = fv.Batch(d, precision=prec, max_patch_size=max(sizes))
    x, toff, tsz = fvtest.to_dev(q), fvtest.to_dev(off), fvtest.to_dev(sz)
    res = []
    for _ in range(2):
        pp = torch.full((n, s), float("nan"), dtype=torch.float64, device="cuda")
        tot = torch.zeros(s, dtype=torch.float64, device="cuda")
        fv.fv_patch_sums(b.h, x, toff, tsz, n, pp, tot)
        res.append((pp.cpu().numpy(), tot.cpu().numpy()))
    assert b.status() == fv.FV_OK
    only = torch.zeros(s, dtype=torch.float64, device="cuda")
    b.totals(x, toff, tsz, only)
    assert np.array_equal(only.cpu().numpy(), res[0][1])
    b.close()
    assert np.array_equal(res[0][0], res[1][0]) and np.array_equal(res[0][1], res[1][1])
    every = [[] for _ in range(s)]
    for i in range(n):
        p = int(sz[i])
        box = q[off[i]:off[i] + (p + 2) ** d * s].reshape((p + 2,) * d + (s,)).astype(np.float64)
        cells = box[(slice(1, p + 1),) * d].reshape(-1, s)
        for k in range(s):
            ref, mag = math.fsum(cells[:, k]), math.fsum(np.abs(cells[:, k]))
            assert abs(res[0][0][i, k] - ref) <= 1e-14 * mag
            every[k].extend(cells[:, k])
    for k in range(s):
        assert abs(res[0][1][k] - math.fsum(every[k])) <= 1e-14 * math.fsum(np.abs(every[k]))
