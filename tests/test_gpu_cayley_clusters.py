"""Cayley step on clusters of CTAs: batches that take each cluster size (one
rotation: the largest cluster; more rotations than resident clusters of 8, 4
and 2), with and without Y, in place, against the oracle.  Bars as in the
other Cayley tests (fp32 products of length n <= 128 against double)."""
import numpy as np
import pytest
import torch

import oracle
from tests.test_gpu_cayley import _case

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(128, 1), (128, 21), (128, 41), (128, 80), (64, 1), (64, 76), (64, 77), (32, 5)])
@pytest.mark.parametrize("iters", [0, 3])
def test_cayley_every_cluster_size(n, batch, iters):
    from paper_2405_16406_gb300 import spinq
    R, g, alpha = _case(n + batch, min(batch, 7), n)
    reps = -(-batch // R.shape[0])
    R, g = (np.ascontiguousarray(np.tile(a, (reps, 1, 1))[:batch]) for a in (R, g))
    Rt, gt = torch.from_numpy(R).cuda(), torch.from_numpy(g).cuda()
    out, y = spinq.cayley_step(Rt, gt, float(alpha), iters, want_y=True)
    k = min(batch, 7)
    ref, yref = oracle.cayley_step(R[:k].astype(np.float64), g[:k].astype(np.float64), float(alpha), iters)
    got, yg = out.cpu().numpy().astype(np.float64), y.cpu().numpy().astype(np.float64)
    for b in range(batch):
        assert np.abs(got[b] - ref[b % k]).max() <= 5e-5
        assert np.abs(yg[b] - yref[b % k]).max() <= 1e-5 * np.abs(yref).max()
    assert np.array_equal(yg, -np.swapaxes(yg, 1, 2))
    spinq.cayley_step(Rt, gt, float(alpha), iters, out=Rt)
    assert torch.equal(Rt, out)
