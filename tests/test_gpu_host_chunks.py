"""The host pipeline's default chunks on ragged batches: the staging that a
handle keeps follows the bytes of the batch, not the size of its first patch,
and the result is the device update's, bitwise."""
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


def run_host(fv, sizes, pinned):
    """Updates 3D FP64 patches of the given sizes on host memory; returns the
    batch's bytes and the device memory the call took."""
    torch = fvtest.torch_cuda()
    n = len(sizes)
    q, off, sz = inputs.random_batch(n, sizes, 3, seed=2)
    b = fv.Batch(3, max_patch_size=int(sz.max()))
    x = fvtest.to_dev(q)
    y = x.clone()
    b.update(x, y, fvtest.to_dev(off), fvtest.to_dev(sz), 0.01, 0.001)
    ref = y.cpu().numpy()
    hin, hout = torch.from_numpy(q), torch.zeros(len(q), dtype=torch.float64)
    if pinned:
        hin, hout = hin.pin_memory(), hout.pin_memory()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    fv.fv_patch_update_host(b.h, hin, hout, off, sz, n, 0.01, 0.001)
    used = free - torch.cuda.mem_get_info()[0]
    mask = fvtest.interior_mask(off, sz, 3, 5, len(q))
    assert b.status() == fv.FV_OK
    assert np.array_equal(hout.numpy()[mask], ref[mask])
    b.close()
    return q.nbytes, used


@pytest.mark.parametrize("first", [1, 8])
def test_staging_follows_the_bytes(fv, first):
    """Three slots of an eighth of the batch each, a patch and the metadata
    (12 B a patch a slot) more, in 2 MB granules."""
    sizes = np.full(3000, 8, dtype=np.int32)
    sizes[0] = first
    total, used = run_host(fv, sizes, True)
    assert used <= 3 * (total / 8 + 40000 + 12 * len(sizes)) + 9 * (4 << 20)


def test_pageable_memory_goes_in_large_chunks(fv):
    """Three slots of the whole batch: its copies do not overlap anyway."""
    total, used = run_host(fv, np.full(1500, 8, dtype=np.int32), False)
    assert used >= 3 * total
