"""The reductions at the edges of their work split: conservation sums for
patch sizes around the lanes and rounds of a warp and patch counts around a
cluster's chunk, against math.fsum per patch (1e-14 of the sum of magnitudes,
the totals' tolerance) and bitwise the same from run to run; the FP64 maximum
eigenvalue where its FP32 bounds cannot decide (ties, states one ulp apart,
velocities far above the sound speed, scales outside the floats' range),
bitwise equal to the update's own maximum of the face wave speeds."""
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


@pytest.mark.parametrize("d,p", [(1, 6), (2, 3), (2, 9), (3, 2), (3, 5)])
@pytest.mark.parametrize("kind", ["random", "uniform", "ulp", "fast", "scales", "rest"])
def test_max_eigenvalue_bitwise(fv, d, p, kind):
    torch = fvtest.torch_cuda()
    s, n = d + 2, 150
    q, off, sz = fvtest.random_batch(n, p, d, 8)
    rng = np.random.default_rng(9)
    for i in range(n):
        c = q[off[i]:off[i] + (p + 2) ** d * s].reshape(-1, s)
        m = len(c)
        rho, u, pr = np.full(m, 1.0 + i / n), np.full((m, d), 0.3), np.full(m, 0.7)
        if kind == "uniform":
            c[:] = inputs.conserved_from_primitive(rho, u, pr)
        elif kind == "ulp":  # pressures a few ulps apart
            pr = pr * (1 + rng.integers(0, 9, m) * 2.0 ** -52)
            c[:] = inputs.conserved_from_primitive(rho, u, pr)
        elif kind == "fast":  # the pressure 1e-9 .. 1e-3 of the energy
            pr = 10.0 ** rng.uniform(-9, -3, m)
            c[:] = inputs.conserved_from_primitive(rho, u * rng.uniform(0.9, 1.1, (m, d)), pr)
        elif kind == "scales":
            c *= 10.0 ** rng.integers(-150, 150)
        elif kind == "rest":
            c[:] = inputs.conserved_from_primitive(rho, 0 * u, pr * rng.uniform(1, 1 + 1e-7, m))
    b = fv.Batch(d, max_patch_size=p)
    x, toff, tsz = fvtest.to_dev(q), fvtest.to_dev(off), fvtest.to_dev(sz)
    y = x.clone()
    lam, per = (torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2))
    gmax, gonly = (torch.zeros(1, dtype=torch.float64, device="cuda") for _ in range(2))
    b.update(x, y, toff, tsz, 1.0, 1e-30, lambda_patch=lam)
    b.max_eigenvalue(x, toff, tsz, 0.4, 1.0, per_patch=per, global_max=gmax)
    b.max_eigenvalue(x, toff, tsz, 0.4, 1.0, global_max=gonly)
    assert b.status() == fv.FV_OK
    assert torch.equal(per, lam) and gmax.item() == lam.max().item() == gonly.item()
    b.close()


@pytest.mark.parametrize("cell", [{"rho": -1.0}, {"rho": 0.0}, {"E": 0.0}, {"E": float("nan")},
                                  {"rho": float("inf")}, {"j": 1e3}])
def test_max_eigenvalue_reports_nonphysical_cells(fv, cell):
    torch = fvtest.torch_cuda()
    d, p, n = 3, 4, 40
    s = d + 2
    q, off, sz = fvtest.random_batch(n, p, d, 8)
    c = q[off[23]:off[23] + (p + 2) ** d * s].reshape(-1, s)
    k = 1 + (p + 2) * (1 + (p + 2) * 2)  # an interior cell
    for name, v in cell.items():
        c[k, {"rho": 0, "j": 1, "E": s - 1}[name]] = v
    b = fv.Batch(d, max_patch_size=p)
    x, toff, tsz = fvtest.to_dev(q), fvtest.to_dev(off), fvtest.to_dev(sz)
    g = torch.zeros(1, dtype=torch.float64, device="cuda")
    for per in (None, torch.zeros(n, dtype=torch.float64, device="cuda")):
        b.max_eigenvalue(x, toff, tsz, 0.4, 1.0, per_patch=per, global_max=g)
        assert b.status() == fv.FV_ERR_NONPHYSICAL
    b.close()
