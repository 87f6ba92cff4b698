"""The fp32 dense update inside the gradient kernels, and the loss from split products, at the sizes where
they end: top layers of 1 to 16 outputs and just above, batches at and past a warp's row, the narrow
kernel's largest batch and one more, tiles with aligned and ragged rows, each update rule.

One step from the oracle's state.  A weight is off by its own rounding and lr (0.1) times the error of its
gradient: chains of at most `in` + B multiply-adds and sums, below 1600 x 2^-24 = 1e-4 of the tensor's
largest, so 1e-5 of the largest weight covers it."""
import numpy as np
import pytest

import oracle
import synthdata
from _gpu_common import built_package, dense_cfgs, dense_segments, max_rel_per_tensor

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rule", ["plain", "heavy_ball", "nesterov"])
@pytest.mark.parametrize("widths,K,B", [((516, 1), 2, 5),            # one output; split logits
                                        ((129, 16), 3, 32),          # the widest narrow layer
                                        ((513, 17), 2, 33),          # past it: the 32-wide tiles
                                        ((260, 36, 3), 2, 1024),     # the narrow kernel's largest batch
                                        ((260, 36, 3), 2, 1025),     # one more
                                        ((1284, 516, 10), 16, 24),   # tiles of 128, ragged at both edges
                                        ((321, 203, 7), 4, 9)])      # rows that are not 16-byte aligned
def test_one_step_matches_the_oracle(widths, K, B, rule):
    P = built_package()
    mom = {"plain": dict(momentum=0.0), "heavy_ball": dict(momentum=0.9, weight_decay=1e-3),
           "nesterov": dict(momentum=0.9, nesterov=True, weight_decay=1e-3)}[rule]
    N = 2 * K * B
    classes = max(widths[-1], 2)
    X, y = synthdata.gaussian_mixture_cached(N, widths[0], classes, 31)
    y = (y % widths[-1]).astype(np.int32)
    g, o = dense_cfgs(P, widths=widths, K=K, B=B, H=2, T=2, N=N, precision=P.FP32, seed=5, **mom)
    rng = np.random.default_rng(9)
    W = np.tile(oracle.init_params(o, oracle.INIT_HE), (K, 1))
    W = W.astype(np.float32)
    U = (0.1 * rng.standard_normal(W.shape)).astype(np.float32) * (mom["momentum"] != 0)
    ctx = P.lsgd_create(g)
    P.lsgd_set_dataset(ctx, X, y)
    for k in range(K):
        P.lsgd_set_params(ctx, k, W[k])
        if mom["momentum"]:
            P.lsgd_set_momentum(ctx, k, U[k])
    P.lsgd_run(ctx, 1)
    Wo, Uo, lo, _ = oracle.run(o, X, y=y, W=W.astype(np.float64), U=U.astype(np.float64), s0=0, n_steps=1)
    segs = dense_segments(widths)
    for k in range(K):
        assert max_rel_per_tensor(P.lsgd_params(ctx, k), Wo[k], segs) <= 1e-5
    np.testing.assert_allclose(P.lsgd_losses(ctx, 1, K)[0], lo[0], rtol=1e-5, atol=1e-6)
    P.lsgd_destroy(ctx)
