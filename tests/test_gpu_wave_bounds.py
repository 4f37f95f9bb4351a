"""The FP32 bounds of an FP64 cell's wave speed at the ends of the range they
accept: heavy cold cells whose squared sound speed lies at the floats'
smallest numbers, light hot ones at their largest, an adiabatic exponent next
to 1 or far above it.  The reduce's maxima equal the update's own (which
evaluates every cell in FP64) bitwise, and a time step hands on the maximum
that a reduce of its result finds."""
import numpy as np
import pytest

from paper_2302_09005_gb300 import inputs
from tests import fvtest

pytestmark = pytest.mark.gpu

# log2 of density and of kinetic energy, log10 of internal / kinetic energy,
# gamma; the velocities vary less than the sound speeds
CORNERS = {"cold": (58, -59, (-5.3, -3), 1.4), "colder": (59.5, -59.5, (-5.4, -4), 1.01),
           "light": (-59, 58, (-5, 1), 1.4), "stiff": (-55, 55, (-3, 1), 1e6),
           "near_one": (30, -30, (-5, -2), 1 + 2.0 ** -40), "plain": (0, 0, (-5, -3), 1.4)}


def cells(rng, m, d, corner):
    lr, lk, (i0, i1), _ = CORNERS[corner]
    rho = 2.0 ** (lr + rng.uniform(-0.05, 0.05, m))
    u = 2.0 ** ((lk + 1 - lr) / 2) * rng.uniform(0.9995, 1.0005, m)
    ke = 0.5 * rho * u * u
    c = np.empty((m, d + 2))
    c[:, 0] = rho
    c[:, 1] = rho * u
    c[:, 2:d + 1] = 0.0
    c[:, d + 1] = ke + ke * 10.0 ** rng.uniform(i0, i1, m)
    return c


@pytest.mark.parametrize("d,p", [(1, 40), (2, 9), (3, 5)])
@pytest.mark.parametrize("corner", sorted(CORNERS))
def test_reduce_at_the_corners(d, p, corner):
    fvtest.ensure_built()
    torch = fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv
    s, n = d + 2, 150
    q, off, sz = fvtest.random_batch(n, p, d, 8)
    rng = np.random.default_rng(4)
    for i in range(n):
        c = q[off[i]:off[i] + (p + 2) ** d * s].reshape(-1, s)
        c[:] = cells(rng, len(c), d, corner)
    b = fv.Batch(d, max_patch_size=p, gamma=CORNERS[corner][3])
    x, toff, tsz = fvtest.to_dev(q), fvtest.to_dev(off), fvtest.to_dev(sz)
    y = x.clone()
    lam, per = (torch.zeros(n, dtype=torch.float64, device="cuda") for _ in range(2))
    gmax = torch.zeros(1, dtype=torch.float64, device="cuda")
    b.update(x, y, toff, tsz, 1.0, 1e-300, lambda_patch=lam)
    b.max_eigenvalue(x, toff, tsz, 0.4, 1.0, per_patch=per)
    assert torch.equal(per, lam)
    b.max_eigenvalue(x, toff, tsz, 0.4, 1.0, global_max=gmax)
    assert gmax.item() == lam.max().item()
    assert b.status() == fv.FV_OK
    b.close()


@pytest.mark.parametrize("d,p", [(2, 9), (3, 5)])
@pytest.mark.parametrize("corner", sorted(CORNERS))
def test_step_hands_on_the_maximum(d, p, corner):
    """Uniform patches, each its own periodic neighbour, are steady; the wave
    speeds ascend, so a block meets its largest last."""
    fvtest.ensure_built()
    torch = fvtest.torch_cuda()
    from paper_2302_09005_gb300 import fv
    s, n = d + 2, 3000
    q, off, sz = fvtest.random_batch(n, p, d, 8)
    every = cells(np.random.default_rng(5), n, d, corner)
    g = CORNERS[corner][3]
    u, e = every[:, 1] / every[:, 0], every[:, d + 1] / every[:, 0]
    every = every[np.argsort(u + np.sqrt(g * (g - 1) * (e - 0.5 * u * u)))]
    for i in range(n):
        q[off[i]:off[i] + (p + 2) ** d * s].reshape(-1, s)[:] = every[i]
    b = fv.Batch(d, max_patch_size=p, gamma=g)
    x, toff, tsz = fvtest.to_dev(q), fvtest.to_dev(off), fvtest.to_dev(sz)
    nbr = fvtest.to_dev(inputs.self_periodic_neighbours(n, d))
    y, z = x.clone(), x.clone()
    lam = torch.zeros(n, dtype=torch.float64, device="cuda")
    b.update(x, y, toff, tsz, 1.0, 1e-300, lambda_patch=lam)
    b.max_eigenvalue(x, toff, tsz, 0.4, 1.0)
    b.time_step(x, y, toff, tsz, nbr, 1.0, 0.4)
    mask = fvtest.interior_mask(off, sz, d, s, len(q))
    assert np.array_equal(y.cpu().numpy()[mask], q[mask])
    b.time_step(y, z, toff, tsz, nbr, 1.0, 0.4)  # its dt comes from the first step's maximum
    assert fv.fv_read_dt(b.h) == 0.4 / (d * lam.max().item())
    assert b.status() == fv.FV_OK
    b.close()
