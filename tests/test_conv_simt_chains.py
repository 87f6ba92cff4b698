"""The fp32 weight gradient's longest chain of roundings: at most 2,048 multiply-adds into one
accumulator whatever the number of workers and the mini-batch."""
import ctypes

import numpy as np
import pytest

from _internal import internal, ptr

LONGEST = 2048  # 64 tiles of 128 pixels, a quarter of each to a thread


def _tiles(B, H, W):
    """128-pixel tiles of B images, 8 to 32 pixels wide (powers of two)."""
    up = lambda v: 1 << (v - 1).bit_length()  # noqa: E731
    tw = min(32, max(8, up(W)))
    th = min(128 // tw, up(H))
    return -(-B // (128 // tw // th)) * -(-W // tw) * -(-H // th)


@pytest.mark.parametrize("H,C", [(32, 16), (16, 32), (8, 64), (35, 12), (1, 4)])
def test_chain_is_bounded(H, C):
    L = internal()
    for K in (1, 2, 5, 16, 31, 64, 500):
        for B in (1, 7, 128, 1024, 8192):
            tiles = _tiles(B, H, H)
            for stride in (1, 2):
                nq = L.t_wgrad_simt_ranges(K, B, H, H, C, C, stride)
                assert 1 <= nq <= tiles
                assert -(-tiles // nq) * 128 // 4 <= LONGEST, (K, B, stride, nq)


@pytest.mark.parametrize("H,W,C,stride,per_sm", [(32, 32, 16, 1, 3), (8, 8, 64, 1, 3), (1, 1, 16, 1, 2),
                                                 (16, 16, 32, 2, 2), (8, 8, 64, 2, 2), (1, 1, 16, 2, 1)])
def test_one_wave_where_the_chains_allow(H, W, C, stride, per_sm):
    # CTAs that an SM holds: its 228 KB of shared memory over two staging buffers of 128 output pixels and
    # the input under them, 64 bytes each, and 1 KB; 192 threads of at most 113 registers leave three
    L = internal()
    blocks = (C // 16) ** 2
    B = 16000 if H == 1 else 4096 // H
    for K in (1, 3, 4):
        wave = per_sm * 152 // (K * blocks)
        assert wave < _tiles(B, H, W) <= 64 * wave
        assert L.t_wgrad_simt_ranges(K, B, H, W, C, C, stride) == wave


@pytest.mark.gpu
def test_equal_terms_at_many_workers():
    # dy = 1, x = 1 + 0.49 / 2048: from 4,096 on an fp32 sum of such terms loses 0.49 / 2048 with every
    # one, so a chain of 8,192 is off by 1.2e-4 of itself.  A chain of n equal terms is off by at most
    # n / 2 x 2^-24: 6.1e-5 at 2,048 (of these, by 4.4e-6).
    import torch

    L = internal()
    G, B, H, C = 64, 128, 16, 32
    v = np.float32(1 + 0.49 / 2048)
    x = torch.full((G, B, H, H, C), float(v), device="cuda")
    dy = torch.ones((G, B, H, H, C), device="cuda")
    nq = L.t_wgrad_simt_ranges(G, B, H, H, C, C, 1)
    part = torch.full((G, nq, C, 3, 3, C), float("nan"), device="cuda")
    assert L.t_wgrad_simt(G, B, H, H, C, C, 1, ptr(x), ptr(dy), ptr(part), ctypes.c_void_p(0)) == 0
    torch.cuda.synchronize()
    got = part.double().sum(1).cpu().numpy()
    seen = np.array([H - 1, H, H - 1])  # rows (and columns) that a tap meets the image in
    want = B * np.outer(seen, seen)[None, None, :, :, None] * float(v)
    assert np.abs(got / want - 1).max() <= LONGEST / 2 * 2.0 ** -24
