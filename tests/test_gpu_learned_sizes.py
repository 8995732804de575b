"""The training and inference kernels where their tiles and vector groups are
ragged: error-vector counts that are not multiples of the group the two-grid
kernel keeps in flight, and grids whose coarse points do not fill a feature tile.
The bounds are those the kernels are held to elsewhere (energies 1e-10, loss
1e-5, gradient 1e-3 in norm, BF16 inference 2e-2)."""
import numpy as np
import pytest

from oracle import learned as ln
from test_gpu_learned import crop_batch, dev, hc, host, params, small_crops

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("size", [7, 15, 31])
@pytest.mark.parametrize("vectors", [1, 5, 6])
def test_twogrid_vector_counts(bmg, size, vectors):
    crops, coefs, vecs = (crop_batch(2, first_seed=1300, vectors=vectors) if size == 31
                          else small_crops(size, 2, seed=60, vectors=vectors))
    theta = params(31, w3_scale=0.2)
    m = bmg.Mlp(theta.astype(np.float32))
    erefs = [ln.two_grid_reference(p, list(v)) for p, v in crops]
    _, _, er = m.twogrid(coefs, vecs)
    assert np.allclose(host(er), np.stack(erefs), rtol=1e-10, atol=0)
    L, g = ln.model_two_grid_loss_grad(theta, [(p, list(v), e) for (p, v), e in zip(crops, erefs)])
    Lg, gg, _ = m.twogrid(coefs, vecs, dev(np.stack(erefs)))
    assert abs(Lg - L) <= 1e-5 * abs(L)
    assert np.linalg.norm(gg - g) <= 1e-3 * np.linalg.norm(g)
    m.close()


@pytest.mark.parametrize("n", [7, 15, 31, 63, 255])
def test_inference_at_ragged_tiles(bmg, n):
    planes = hc(n, 90 + n, block=2 if n < 31 else 8)
    theta = params(33, w3_scale=0.3)
    m = bmg.Mlp(theta.astype(np.float32))
    got = host(m.infer(dev(planes)))
    want, _ = ln.forward(theta, ln.features(planes))
    assert np.linalg.norm(got - want) <= 2e-2 * np.linalg.norm(want)
    m.close()


@pytest.mark.parametrize("n", [7, 15, 127])
def test_features_at_ragged_tiles(bmg, n):
    planes = hc(n, 95 + n, block=2 if n < 31 else 8)
    assert np.array_equal(host(bmg.mlp_features(dev(planes))), ln.features(planes).astype(np.float32))
