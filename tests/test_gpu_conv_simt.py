"""The fp32-core convolutions against the oracle: the gradient of one ResNet step at geometries that
cut their tiles (images narrower, wider and taller than a tile, odd sizes under stride 2, channel
counts that are no multiple of the 16-channel block or of 4, a batch that leaves a partial tile, few
CTAs and many)."""
import numpy as np
import pytest

import oracle
from _gpu_common import built_package, rel_l2
from test_gpu_resnet import resnet_cfgs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("hwc,base,B,K", [((32, 32, 3), 16, 6, 2), ((9, 7, 5), 12, 5, 3),
                                          ((35, 41, 16), 8, 3, 1), ((2, 3, 1), 4, 40, 2),
                                          ((16, 8, 64), 4, 7, 1),
                                          ((16, 16, 3), 16, 320, 1)])  # more than two CTAs per SM
def test_fp32_step_gradient(hwc, base, B, K):
    P = built_package()
    N, C = max(K * B, 64), 5
    rng = np.random.default_rng(base + B)
    X = rng.standard_normal((N, int(np.prod(hwc)))).astype(np.float32)
    y = rng.integers(0, C, N).astype(np.int32)
    g, o = resnet_cfgs(P, hwc=hwc, base=base, blocks=1, classes=C, K=K, B=B, H=8, T=8, N=N,
                       precision=P.FP32, base_lr=0.01, momentum=0.9, seed=5)
    ctx = P.lsgd_create(g)
    P.lsgd_set_dataset(ctx, X, y)
    w0 = oracle.init_params(o).astype(np.float32)
    P.lsgd_set_params(ctx, -1, w0)
    P.lsgd_local_step(ctx)
    _, U, lo, _ = oracle.run(o, X, y=y, W=np.tile(w0.astype(np.float64), (K, 1)), n_steps=1)
    np.testing.assert_allclose(P.lsgd_losses(ctx, 1, K)[0], lo[0], rtol=1e-5, atol=1e-6)
    # after one step from zero momentum u is the gradient.  A product's fp32 sums (at most a few
    # thousand terms, about sqrt(n) 2^-24 = 4e-6 of their size) pass through at most 14 further
    # products: 6e-5.  A tap, halo or channel read wrongly is off by the size of a term, > 1e-3.
    for k in range(K):
        assert rel_l2(P.lsgd_momentum(ctx, k), U[k]) <= 1e-4
    P.lsgd_destroy(ctx)
