"""Learned interpolation outside the range that trained networks stay in: logits
so far apart that their exponentials' ratio leaves FP64, on operators with edge
points that have no coupling to one of their sides, whose share is then exactly
0 or 1 (the bound is that of the weights elsewhere, 1e-14 of the largest); and
two-grid crops scaled by powers of two towards the ends of FP64, whose energies
scale with them bit for bit, while loss and gradient, which are relative to the
scaled reference energies, stay the same bits."""
import numpy as np
import pytest

import torch

import workloads as w
from oracle import learned as ln
from test_gpu_learned import crop_batch, dev, host, params, small_crops

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


@pytest.mark.parametrize("size", [7, 15, 31])
def test_twogrid_scales_with_the_operator(bmg, size):
    _, coefs, vecs = crop_batch(2, first_seed=1400) if size == 31 else small_crops(size, 2, seed=80)
    m = bmg.Mlp(params(31, w3_scale=0.2).astype(np.float32))
    _, _, er = m.twogrid(coefs, vecs)
    loss, grad, en = m.twogrid(coefs, vecs, er)
    assert np.isfinite(host(en)).all() and np.isfinite(grad).all()
    for k in (-800, -540, 540, 800):
        s = 2.0 ** k
        _, _, ers = m.twogrid(coefs * s, vecs)
        assert torch.equal(ers, er * s), k
        losss, grads, ens = m.twogrid(coefs * s, vecs, ers)
        assert torch.equal(ens, en * s) and losss == loss and np.array_equal(grads, grad), k
    m.close()
