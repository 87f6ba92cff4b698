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


CASES = pytest.mark.parametrize("widths,K,B", [
    ((516, 1), 2, 5),            # one output; split logits
    ((129, 16), 3, 32),          # the widest narrow layer
    ((513, 17), 2, 33),          # past it: the 32-wide tiles
    ((260, 36, 3), 2, 1024),     # the narrow kernel's largest batch
    ((260, 36, 3), 2, 1025),     # one more
    ((1284, 516, 10), 16, 24),   # tiles of 128, ragged at both edges
    ((321, 203, 7), 4, 9)])      # rows that are not 16-byte aligned
RULES = {"plain": dict(momentum=0.0), "heavy_ball": dict(momentum=0.9, weight_decay=1e-3),
         "nesterov": dict(momentum=0.9, nesterov=True, weight_decay=1e-3)}


@pytest.mark.parametrize("rule", list(RULES))
@CASES
def test_one_step_matches_the_oracle(widths, K, B, rule):
    P = built_package()
    mom = RULES[rule]
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
        if mom["momentum"]:  # u = 0.9 U + gradient, the largest of a tensor at least half the gradient's
            assert max_rel_per_tensor(P.lsgd_momentum(ctx, k), Uo[k], segs) <= 2e-4
    np.testing.assert_allclose(P.lsgd_losses(ctx, 1, K)[0], lo[0], rtol=1e-5, atol=1e-6)
    P.lsgd_destroy(ctx)


@pytest.mark.parametrize("rule", list(RULES))
@CASES
def test_one_step_has_the_bits_of_the_stand_alone_update(widths, K, B, rule):
    # a step from zero momentum without decay leaves the gradient itself as the momentum; the stand-alone
    # update on it and the case's own state is then the step's result, bit for bit
    import torch

    P = built_package()
    mom, N = RULES[rule], 2 * K * B
    X, y = synthdata.gaussian_mixture_cached(N, widths[0], max(widths[-1], 2), 31)
    y = (y % widths[-1]).astype(np.int32)
    rng = np.random.default_rng(10)
    _, o = dense_cfgs(P, widths=widths, K=K, B=B, H=2, T=2, N=N, precision=P.FP32, seed=5)
    W = np.tile(oracle.init_params(o, oracle.INIT_HE), (K, 1)).astype(np.float32)
    U = (0.1 * rng.standard_normal(W.shape)).astype(np.float32)

    def step(U0, **kw):
        g, _ = dense_cfgs(P, widths=widths, K=K, B=B, H=2, T=2, N=N, precision=P.FP32, seed=5, **kw)
        ctx = P.lsgd_create(g)
        P.lsgd_set_dataset(ctx, X, y)
        for k in range(K):
            P.lsgd_set_params(ctx, k, W[k])
            if kw["momentum"] and U0 is not None:
                P.lsgd_set_momentum(ctx, k, U0[k])
        P.lsgd_run(ctx, 1)
        out = [np.stack([f(ctx, k) for k in range(K)]) for f in (P.lsgd_params, P.lsgd_momentum)]
        P.lsgd_destroy(ctx)
        return out

    G = step(None, momentum=0.9)[1]
    W1, U1 = step(U, **mom)
    n = W.size + (-W.size) % 4
    w, u, g = (torch.zeros(n, device="cuda") for _ in range(3))
    for t, a in ((w, W), (u, U), (g, G)):
        t[:W.size] = torch.from_numpy(a.reshape(-1)).cuda()
    has_u = mom["momentum"] != 0
    P.lsgd_sgd_update(w, u if has_u else None, g, None, n, 0.1, mom["momentum"], mom.get("nesterov", False),
                      mom.get("weight_decay", 0.0))
    assert np.array_equal(w[:W.size].cpu().numpy().reshape(W.shape), W1)
    if has_u:
        assert np.array_equal(u[:W.size].cpu().numpy().reshape(W.shape), U1)


def test_no_gradient_array():
    # the gradients are never in memory: one array of parameters, and the activations, are all that is asked for
    import torch

    P = built_package()
    asked = []

    def _alloc(user, nbytes, stream):
        asked.append(int(nbytes))
        return torch.cuda.caching_allocator_alloc(int(nbytes), 0, stream)

    def _free(user, p, stream):
        torch.cuda.caching_allocator_delete(p)

    a = P.Allocator(P.ALLOC_FN(_alloc), P.FREE_FN(_free), None)
    K, widths = 3, (2048, 2048, 10)
    g, _ = dense_cfgs(P, widths=widths, K=K, B=4, H=1, T=1, N=64, precision=P.FP32)
    ctx = P.lsgd_create(g, allocator=a)
    params = 4 * K * sum(i * o for i, o in zip(widths[:-1], widths[1:]))
    assert sum(n >= params for n in asked) == 1
    P.lsgd_destroy(ctx)
