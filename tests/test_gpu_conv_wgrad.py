"""The convolution weight-gradient kernel (tcgen05, taps as shifted views of one input strip) against
an fp64 evaluation of its definition on the same bf16 operands:
    dW[g][co][kh][kw][ci] = sum over b, oy, ox of dy[g][b][oy][ox][co] x[g][b][s oy + kh - 1][s ox + kw - 1][ci]
(3x3 kernel, zero padding 1, stride s).  Every ResNet-20 shape (16 / 32 / 64 channels, both
strides, 32 / 16 / 8 wide outputs), several groups and several CTAs per group.  Error measure:
|dW - dW64| / (sum |dy| |x|) elementwise, the fp32 accumulation bound's scale; a wrong tap,
channel or halo row moves an element by ~1 / sqrt(terms) of that scale, far above the bar."""
import numpy as np
import pytest

from _gpu_common import built_package

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch

    assert torch.cuda.is_available()
    return built_package()


def _reference(x, dy, stride):
    """fp64 weight gradient from the definition: pad the input, slice each tap's shifted view."""
    G, B, Hin, Win, Cin = x.shape
    Hout, Wout = dy.shape[2], dy.shape[3]
    xp = np.zeros((G, B, Hin + 2, Win + 2, Cin))
    xp[:, :, 1:Hin + 1, 1:Win + 1, :] = x
    dW = np.zeros((G, dy.shape[4], 3, 3, Cin))
    scale = np.zeros_like(dW)
    for kh in range(3):
        for kw in range(3):
            # input pixel (s oy + kh - 1, s ox + kw - 1) = padded pixel (s oy + kh, s ox + kw)
            v = xp[:, :, kh:kh + stride * Hout:stride, kw:kw + stride * Wout:stride, :]
            dW[:, :, kh, kw, :] = np.einsum("gbhwo,gbhwi->goi", dy, v)
            scale[:, :, kh, kw, :] = np.einsum("gbhwo,gbhwi->goi", np.abs(dy), np.abs(v))
    return dW, scale


SHAPES = [  # (G, B, Hout, Wout, Cin, Cout, stride)
    (2, 6, 32, 32, 16, 16, 1),
    (3, 4, 16, 16, 16, 32, 2),
    (2, 5, 16, 16, 32, 32, 1),
    (2, 6, 8, 8, 32, 64, 2),
    (3, 7, 8, 8, 64, 64, 1),
    (1, 3, 8, 16, 64, 48, 1),
    (4, 1, 8, 8, 16, 16, 1),
]


@pytest.mark.parametrize("shape", SHAPES)
def test_conv_wgrad_matches_fp64(P, shape):
    import torch

    G, B, Hout, Wout, Cin, Cout, s = shape
    gen = torch.Generator(device="cuda").manual_seed(sum(shape))
    x = torch.randn((G, B, s * Hout, s * Wout, Cin), device="cuda", generator=gen).to(torch.bfloat16)
    dy = torch.randn((G, B, Hout, Wout, Cout), device="cuda", generator=gen).to(torch.bfloat16)
    dW = torch.full((G, Cout, 3, 3, Cin), float("nan"), device="cuda")
    P.lsgd_conv_wgrad_bf16(x, dy, dW, G, B, Hout, Wout, Cin, Cout, s)
    torch.cuda.synchronize()
    want, scale = _reference(x.float().cpu().numpy().astype(np.float64),
                             dy.float().cpu().numpy().astype(np.float64), s)
    got = dW.cpu().numpy().astype(np.float64)
    err = np.abs(got - want) / np.maximum(scale, 1e-30)  # a tap that never meets the image: exactly zero
    assert np.isfinite(got).all()
    assert err.max() <= 1e-5, err.max()


def test_conv_wgrad_is_deterministic(P):
    import torch

    G, B, Hout, Wout, Cin, Cout, s = 2, 8, 32, 32, 16, 32, 1
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((G, B, Hout, Wout, Cin), device="cuda", generator=gen).to(torch.bfloat16)
    dy = torch.randn((G, B, Hout, Wout, Cout), device="cuda", generator=gen).to(torch.bfloat16)
    outs = []
    for _ in range(2):
        dW = torch.empty((G, Cout, 3, 3, Cin), device="cuda")
        P.lsgd_conv_wgrad_bf16(x, dy, dW, G, B, Hout, Wout, Cin, Cout, s)
        outs.append(dW.cpu())
    assert torch.equal(outs[0], outs[1])


def test_conv_wgrad_rejects_unsupported_shapes(P):
    import torch

    x = torch.zeros((1, 1, 8, 8, 16), device="cuda", dtype=torch.bfloat16)
    dy = torch.zeros((1, 1, 8, 8, 16), device="cuda", dtype=torch.bfloat16)
    dW = torch.zeros((1, 16, 3, 3, 16), device="cuda")
    for bad in [dict(Cin=8), dict(Cout=8), dict(Cout=80), dict(stride=3), dict(Hout=4, Wout=4),
                dict(Wout=12)]:
        kw = dict(G=1, B=1, Hout=8, Wout=8, Cin=16, Cout=16, stride=1)
        kw.update(bad)
        with pytest.raises(P.LsgdError):
            P.lsgd_conv_wgrad_bf16(x, dy, dW, **kw)


@pytest.mark.parametrize("shape", [(2, 3, 2, 64, 16, 16, 1), (1, 2, 4, 64, 64, 64, 2),   # widest rows
                                   (2, 3, 2, 32, 32, 16, 1), (1, 5, 4, 16, 64, 32, 2),   # 64-pixel tiles
                                   (3, 2, 16, 8, 16, 48, 1), (1, 9, 16, 8, 32, 64, 2),   # two rows per step
                                   # narrower than 8: tiles of 64 and of 128 pixels down the columns
                                   (2, 3, 16, 4, 16, 32, 1), (1, 2, 32, 2, 32, 16, 2), (3, 5, 64, 1, 64, 48, 1),
                                   (2, 3, 128, 1, 32, 32, 1), (1, 3, 128, 1, 16, 16, 2), (2, 7, 64, 2, 16, 64, 1),
                                   (1, 2, 96, 2, 32, 16, 2), (1, 3, 160, 4, 64, 64, 1), (2, 2, 32, 4, 64, 32, 2),
                                   (1, 5, 48, 4, 32, 48, 2), (20, 9, 64, 1, 64, 64, 2)])
def test_conv_wgrad_tile_edges(P, shape):
    test_conv_wgrad_matches_fp64(P, shape)


def test_conv_wgrad_of_narrow_outputs_runs_on_the_tensor_cores(P):
    # the same pixels, channels and products as 64 x 1, 16 x 4 and 8 x 8 images.  Narrow rows cost more
    # loads per tile, at most ten for an 8-pixel row's two; the fp32 cores take fifty times the 8 x 8 time.
    import torch

    def us(Hout, Wout, G=16, B=128, C=64):
        x = torch.ones((G, B, Hout, Wout, C), device="cuda", dtype=torch.bfloat16)
        dW = torch.empty((G, C, 3, 3, C), device="cuda")
        times = []
        for _ in range(5):
            a, b = (torch.cuda.Event(enable_timing=True) for _ in range(2))
            a.record()
            for _ in range(10):
                P.lsgd_conv_wgrad_bf16(x, x, dW, G, B, Hout, Wout, C, C, 1)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b) * 100)
        return min(times)

    wide = us(8, 8)
    assert us(64, 1) <= 5 * wide
    assert us(16, 4) <= 5 * wide
