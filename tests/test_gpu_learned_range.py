"""Learned interpolation outside the range that trained networks stay in: logits
so far apart that their exponentials' ratio leaves FP64, on operators with edge
points that have no coupling to one of their sides, whose share is then exactly
0 or 1.  The bound is that of the weights elsewhere, 1e-14 of the largest."""
import numpy as np
import pytest

import torch

import workloads as w
from oracle import learned as ln
from test_gpu_learned import dev, host

pytestmark = pytest.mark.gpu


def cut_planes(n, columns, rows):
    """A lognormal operator without the couplings from columns (rows) k to k - 1."""
    planes = w.fe9_from_cells(w.lognormal_cells(n, 1.0, 4.0, 40 + n))
    for i in columns:
        planes[(1, 3, 4), :, i] = 0.0
    for j in rows:
        planes[(2, 3), j, :] = 0.0
        planes[4, j - 1, :] = 0.0
    return planes


@pytest.mark.parametrize("n", [7, 63])
@pytest.mark.parametrize("span", [50.0, 299.0, 301.0, 400.0, 700.0])
def test_weights_of_distant_logits(bmg, n, span):
    # cuts on either side of an odd line: no coupling west (south) of it, none east (north)
    planes = cut_planes(n, (3, n - 1), (3, n - 1))
    nc = (n - 1) // 2
    delta = np.sign(w.normal(7, nc * nc * 4).reshape(nc * nc, 4)) * span
    want = ln.learned_interp(planes, delta)
    assert np.isfinite(want).all()
    got = host(bmg.learned_interp(dev(planes), dev(delta, torch.float32)))
    assert np.abs(got - want).max() <= 1e-14 * np.abs(want).max()
