"""The denoiser's weight gradients at the edges of their row segments: widths that are no multiple
of the 16 voxels of one product, rows of more than one segment, one row per plane, planes
outside the window; against the numpy oracle at the GPU's BF16 rounding points.  Tolerance 2e-2
of the largest entry, as for the whole gradient: a BF16 rounding of an activation that the
FP32 summation order flips moves single products by 2^-8."""
import numpy as np
import pytest

from oracle import denoise_ref as D
from tests.test_denoise_gpu import _oracle_forward, _to_gpu

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def G():
    import torch
    if not torch.cuda.is_available():
        pytest.fail("GPU tests need a CUDA device")
    from paper_2509_16793_gb300 import build, gempic
    build.build()
    return gempic


@pytest.mark.parametrize("shape", [(7, 1, 40), (3, 3, 130), (9, 5, 17), (4, 2, 8), (1, 4, 128),
                                   (5, 2, 300)])
def test_weight_gradient_at_segment_edges(G, shape):
    nz, ny, nx = shape
    rng = np.random.default_rng(sum(shape))
    scale = 0.05
    j, t = (np.asarray(rng.standard_normal((nz, ny, nx, 3)) * scale, np.float32).astype(np.float64)
            for _ in range(2))
    P = D.init_params(seed=7, scale3=1.0)
    with G.Denoiser(G.denoiser_params_to_vector(P), scale) as d:
        loss, g = d.grad(_to_gpu(j), _to_gpu(t))
        again = d.grad(_to_gpu(j), _to_gpu(t))[1]
    assert np.array_equal(g, again)                      # partial sums added in a fixed order
    Q, x0, h1, h2, r = _oracle_forward(P, j, scale)
    e = (j - t) / scale + r
    dr = D.to_bf16(2.0 * e / e.size)
    dh2, gW3, gb3 = D.conv3d_backward(h2, Q["W3"], dr)
    dh2 = D.to_bf16(dh2 * (h2 > 0))
    dh1, gW2, gb2 = D.conv3d_backward(h1, Q["W2"], dh2)
    dh1 = D.to_bf16(dh1 * (h1 > 0))
    _, gW1, gb1 = D.conv3d_backward(x0, Q["W1"], dh1)
    gP = G.denoiser_vector_to_params(g)
    for name, want in (("W3", gW3), ("b3", gb3), ("W2", gW2), ("b2", gb2), ("W1", gW1), ("b1", gb1)):
        err = np.abs(gP[name] - want).max() / np.abs(want).max()
        assert err < 2e-2, (name, err)
