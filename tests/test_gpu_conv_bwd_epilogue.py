"""The super-pixel convolution's BatchNorm-backward epilogue on its own: what it stores,

  g = (dx + shortcut) (mask > 0),   shortcut = sc_dout (sc_out > 0) at the pixels on the block's stride grid,

with dx the data gradient of the 3x3 convolution, and the sums over the pixels of g and g (y - mean) rstd per
replica and channel.  Operands are small whole numbers (rstd powers of two), so that every product and every
partial sum, in any order, is a whole number below 2^24: the results have to be exact."""
import ctypes

import numpy as np
import pytest

from _internal import internal, ptr
from test_gpu_conv_tc import _dgrad64

pytestmark = pytest.mark.gpu

# (G, B, Hin, Win, Cin = N, Cout = ck, stride): tiles of 16 image rows where G B (rows / 16) >= 304, else of 8;
# more tiles than CTAs in unequal shares where G does not divide the 152 SMs or the tiles
SHAPES = [(3, 3, 32, 32, 16, 16, 1), (5, 61, 32, 32, 16, 16, 1),   # 16 channels
          (2, 5, 16, 16, 32, 32, 1), (16, 20, 16, 16, 32, 32, 1),  # 32
          (2, 6, 8, 8, 64, 64, 1), (7, 45, 8, 8, 64, 64, 1),       # 64: image rows of one tile
          (1, 2, 24, 32, 16, 16, 1),                               # three tiles of eight rows
          (2, 5, 32, 32, 16, 32, 2), (16, 20, 32, 32, 16, 32, 2),  # parity phases, two segments
          (3, 6, 16, 16, 32, 64, 2), (7, 45, 16, 16, 32, 64, 2)]


@pytest.mark.parametrize("shortcut", [False, True])
@pytest.mark.parametrize("shape", SHAPES)
def test_stored_gradient_and_sums(shape, shortcut):
    import torch

    L = internal()
    G, B, H, W, N, ck, s = shape
    rng = np.random.default_rng(sum(shape))
    ints = lambda r, *d: rng.integers(-r, r + 1, d).astype(np.float64)  # noqa: E731
    dy, w = ints(2, G, B, H // s, W // s, ck), ints(2, G, ck, 3, 3, N)
    mask, y, mean = ints(1, G, B, H, W, N), ints(3, G, B, H, W, N), ints(1, G, N)
    rstd = 2.0 ** rng.integers(-2, 2, (G, N))
    want = _dgrad64(dy, w, s, H, W)[0]
    sd, so = ints(50, G, B, H // s, W // s, ck), ints(1, G, B, H // s, W // s, ck)
    if shortcut:
        want[:, :, ::s, ::s] += (sd * (so > 0))[..., :N]
    want *= mask > 0
    sums = np.stack([want.sum((1, 2, 3)), (want * (y - mean[:, None, None, None])).sum((1, 2, 3)) * rstd], -1)

    # the kernel's weights: [Cin][tap][Cout] of the flipped taps, or of the four parity phases' taps
    wt = w.transpose(0, 4, 2, 3, 1)
    if s == 1:
        packed = wt[:, :, ::-1, ::-1]
    else:
        packed = np.zeros((4,) + wt.shape)
        for ph in range(4):
            for th in range(3):
                for tw in range(3):
                    kh, kw = (ph >> 1) + 1 - 2 * (th - 1), (ph & 1) + 1 - 2 * (tw - 1)
                    if 0 <= kh <= 2 and 0 <= kw <= 2:
                        packed[ph, :, :, th, tw] = wt[:, :, kh, kw]
    dev = lambda a, t: torch.from_numpy(np.ascontiguousarray(a)).to("cuda", t)  # noqa: E731
    bf, f = torch.bfloat16, torch.float32
    t = dict(dy=dev(dy, bf), w=dev(packed, bf), mask=dev(mask, bf), y=dev(y, f), mean=dev(mean, f),
             rstd=dev(rstd, f), sd=dev(sd, f), so=dev(so, bf))
    out = torch.full((G, B, H, W, N), float("nan"), device="cuda")

    def call(part):
        return L.t_conv_sp_bwd(G, B, H // s, W // s, ck, N, int(s == 2), ptr(t["dy"]), ptr(t["w"]), ptr(out),
                               ptr(t["mask"]), ptr(t["y"]), ptr(t["mean"]), ptr(t["rstd"]),
                               ptr(t["sd"] if shortcut else None), ptr(t["so"] if shortcut else None), ck, s,
                               part, ctypes.c_void_p(torch.cuda.current_stream().cuda_stream))

    n = call(ctypes.c_void_p(0))
    assert n > 0
    part = torch.full((G, n, N, 2), float("nan"), device="cuda")
    assert call(ptr(part)) == n
    torch.cuda.synchronize()
    np.testing.assert_array_equal(out.double().cpu().numpy(), want)
    np.testing.assert_array_equal(part.double().sum(1).cpu().numpy(), sums)
