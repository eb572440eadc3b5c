"""Convolutions whose taps share one load of the activation (spmm_halo.cu), at the edges of its tiles: one, two and four
images a tile, 224 and 256 pixels, ragged in x, y, images and output channels, several slabs of channels and CTA tiles of rows,
weight tiles that stay and that do not.

Reference: the same layer's product with [channels, pixels] results, which the taps' own loads compute (and the oracle checks
elsewhere), and the oracle's convolution of one image's top strip.  Both round one fp32 sum of at most t products to bf16; two orders of
such a sum differ by at most 2 t * 2^-23 * sum |w x|, their bf16 roundings by at most 2^-7 of the value."""
import numpy as np
import pytest

import oracle
from helpers import bf16_dev, gpu_layer, oracle_layer, to_dev, y_to_f64
from test_gpu_conv import conv_inputs

pytestmark = pytest.mark.gpu

CASES = [
    # s_out, kh, kw, pad, c, b, h, w, n, m, bm, keep, tile, whether the weight tiles stay
    (64, 3, 3, 1, 64, 20, 84, 80, 2, 4, 64, 0.4, 224, True),        # one CTA tile of rows, weight tiles stay
    (64, 3, 3, 1, 64, 26, 64, 96, 3, 4, 64, 0.9, 256, False),        # 64-pixel columns: 256 pixels cover less; nine blocks, dense tiles
    (200, 3, 3, 1, 128, 27, 28, 28, 1, 4, 64, 0.5, 224, False),      # ragged in x and in the channels, two slabs, two CTA tiles of rows
    (256, 3, 3, 1, 192, 75, 14, 14, 2, 4, 32, 0.3, 224, False),      # two images a tile, an odd number of them, three slabs
    (264, 3, 3, 1, 64, 203, 7, 7, 4, 8, 128, 0.6, 224, False),       # four images a tile, dense tiles, three CTA tiles of rows
    (96, 5, 3, 2, 64, 40, 33, 57, 2, 4, 32, 0.8, 224, False),        # odd sizes, border of four rows and two columns, images of four
    (160, 3, 3, 0, 64, 17, 34, 66, 2, 8, 32, 0.4, 256, False),       # no padding, 32-pixel columns
    (256, 3, 3, 1, 64, 12, 56, 56, 2, 4, 64, 0.9, 256, False),       # 256 pixels of four images, one accumulator
    (200, 3, 3, 1, 64, 5, 9, 8, 1, 4, 128, 0.34, 64, False),  # few tiles: 64 pixels, ragged in y and in the channels
    (96, 3, 3, 1, 128, 3, 19, 22, 3, 4, 64, 0.5, 64, False),  # the same with dense tiles, odd sizes
    (256, 3, 3, 1, 128, 31, 14, 14, 4, 8, 64, 0.2, 128, False),   # 128 pixels, dense tiles, an odd number of images
    (235, 3, 3, 1, 128, 6, 7, 7, 1, 4, 128, 0.3, 64, False),  # 235 channels: stored pixel by pixel
    (100, 3, 3, 1, 128, 80, 28, 27, 2, 4, 32, 0.5, 224, False),   # 100 channels, several images, ragged in x
    (256, 1, 1, 0, 64, 16, 56, 50, 2, 4, 64, 1.0, 224, False),    # 1x1: no border, ragged in x
    (72, 1, 1, 0, 192, 50, 45, 41, 1, 8, 32, 0.7, 224, True),
    (448, 3, 3, 1, 256, 30, 28, 28, 4, 8, 32, 0.59, 224, False),  # dense tiles, four waves where the other kernel has three
    (320, 1, 1, 0, 128, 6, 28, 28, 1, 8, 64, 1.0, 128, False),    # two blocks, 256-pixel tiles in the other kernel
]


def layer_and_input(s_out, kh, kw, c, b, h, w, n, m, bm, keep, seed):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    wt, sal, act = conv_inputs(s_out, kh, kw, c, b, h, w, seed=seed)
    L = gpu_layer(B, torch, wt, sal, n, m, bm, 64, keep)
    bias = np.random.default_rng(seed).standard_normal(s_out).astype(np.float32)
    L.set_epilogue(to_dev(bias, torch), relu=True)
    return torch, B, L, wt, sal, act, bias


@pytest.mark.parametrize("s_out,kh,kw,pad,c,b,h,w,n,m,bm,keep,tile,stay", CASES)
def test_convolution(s_out, kh, kw, pad, c, b, h, w, n, m, bm, keep, tile, stay):
    torch, B, L, wt, sal, act, bias = layer_and_input(s_out, kh, kw, c, b, h, w, n, m, bm, keep, s_out + h)
    mk, vals, idx, wd, _ = oracle_layer(wt, sal, n, m, bm, 64, keep)
    x = bf16_dev(act, torch)
    ho, wo = h + 2 * pad - kh + 1, w + 2 * pad - kw + 1
    buf = torch.full((b * ho * wo * s_out + 64,), 7.0, dtype=torch.bfloat16, device="cuda")
    y = buf[:b * ho * wo * s_out].view(b, ho, wo, s_out)
    L.spmm_conv(x, kh, kw, pad, y=y, nhwc_out=True)
    torch.cuda.synchronize()
    info = L.last_launch()
    assert L.device_status() == 0 and info["tile_cols"] == tile and info["epilogue_warps"] == 16
    assert (L.last_resident_bytes() > 0) == stay
    other = L.spmm_conv(x, kh, kw, pad)                         # [channels, pixels]: every tap loads its own pixels
    assert L.last_launch()["tile_cols"] in (128, 256) and L.last_launch()["stages"] >= 2
    terms = mk.kkeep * 64 * n // m + 1
    mag = float(np.abs(wd).max()) * float(x.abs().max()) * terms
    a, r = y.reshape(-1, s_out).t().double(), other.double()
    assert bool(((a - r).abs() <= 2.0 ** -7 * r.abs() + 2 * terms * 2.0 ** -23 * mag).all())
    rows = min(h, 8)
    ref = oracle.bias_relu(oracle.conv_fp64(wd, kh, kw, np.ascontiguousarray(act[-1:, :rows]), pad), bias, True).reshape(s_out, -1, wo)
    inner = rows - kh + pad + 1                                 # output rows whose window lies in the strip
    got = y_to_f64(y[-1, :inner].reshape(-1, s_out), torch).T.reshape(s_out, inner, wo)
    assert np.all(np.abs(got - ref[:, :inner]) <= 2.0 ** -8 * np.abs(ref[:, :inner]) + terms * 2.0 ** -23 * mag)
    assert torch.all(buf[b * ho * wo * s_out:] == 7.0)
    L.close()


@pytest.mark.parametrize("s_out,kh,c,b,h,w,n,m,bm,keep", [
    (384, 3, 512, 1, 112, 112, 1, 4, 64, 0.69),      # two waves of tiles here, one in the kernel that loads the pixels of each tap
    (128, 3, 128, 40, 28, 28, 1, 4, 64, 0.59),
    (448, 3, 512, 5, 55, 57, 2, 8, 64, 0.9),         # three and two
    (448, 1, 64, 4, 28, 28, 2, 8, 128, 1.0),         # one wave, one block
])
def test_convolutions_that_sharing_loads_would_slow_down(s_out, kh, c, b, h, w, n, m, bm, keep):
    torch, B, L, wt, sal, act, bias = layer_and_input(s_out, kh, kh, c, b, h, w, n, m, bm, keep, 1)
    x = bf16_dev(act, torch)
    y = L.spmm_conv(x, kh, kh, kh // 2, nhwc_out=True)
    taken = L.last_launch()
    L.set_stage_blocks(1)                                       # (one tap a load)
    other = L.spmm_conv(x, kh, kh, kh // 2, nhwc_out=True)
    torch.cuda.synchronize()
    forced = L.last_launch()
    assert all(taken[f] == forced[f] for f in ("tile_cols", "epilogue_warps", "accumulators", "ctas"))
    assert L.device_status() == 0 and torch.equal(y, other)
    L.close()


@pytest.mark.parametrize("y_dtype", [0, 1])
@pytest.mark.parametrize("s_out,ldy,b,h,w", [
    (100, 104, 20, 28, 28), (100, 128, 1, 28, 28), (235, 240, 6, 7, 7), (45, 48, 4, 56, 56), (45, 48, 1, 14, 14), (45, 48, 40, 112, 112),
    (30, 32, 3, 56, 56), (130, 144, 9, 28, 28), (67, 68, 2, 19, 21), (96, 104, 5, 28, 28),
])
def test_what_lies_behind_the_channels_of_a_pixel_stays(s_out, ldy, b, h, w, y_dtype):
    """Pixels further apart than their channels, in both convolution kernels (fp32 results leave by the older one)."""
    torch, B, L, wt, sal, act, bias = layer_and_input(s_out, 3, 3, 64, b, h, w, 2, 4, 32, 0.6, s_out + h)
    x = bf16_dev(act, torch)
    buf = torch.full((b, h, w, ldy), 7.0, dtype=torch.float32 if y_dtype else torch.bfloat16, device="cuda")
    terms = 5 * 64 * 2 // 4 + 1                                 # five of nine blocks, and the bias
    mag = terms * max(1.0, float(x.abs().max())) * float(bf16_dev(wt, torch).abs().max()) + float(np.abs(bias).max())
    for stage_blocks in (0, 1):                                 # (a bound on the blocks of a stage: the older kernel)
        buf.fill_(7.0)
        L.set_stage_blocks(stage_blocks)
        L.spmm_conv(x, 3, 3, 1, y=buf[..., :s_out], y_dtype=y_dtype, nhwc_out=True)
        torch.cuda.synchronize()
        assert L.device_status() == 0 and bool((buf[..., s_out:] == 7.0).all())
        other = L.spmm_conv(x, 3, 3, 1, y_dtype=1).t().reshape(b, h, w, s_out)
        order = 2 * terms * 2.0 ** -23 * mag                    # two orders of an fp32 sum
        assert bool(((buf[..., :s_out].float() - other).abs() <= (0.0 if y_dtype else 2.0 ** -8) * other.abs() + order).all())
    L.close()


def test_a_wait_that_runs_out_is_reported():
    torch, B, L, wt, sal, act, bias = layer_and_input(64, 3, 3, 64, 20, 84, 80, 2, 4, 64, 0.4, 3)
    x = bf16_dev(act, torch)
    want = L.spmm_conv(x, 3, 3, 1, nhwc_out=True)
    L.set_tuning(wait_limit_cycles=2_000_000, skip_fill=1)      # every CTA's second load of the activation is left out
    L.spmm_conv(x, 3, 3, 1, nhwc_out=True)
    torch.cuda.synchronize()
    assert L.last_launch()["tile_cols"] == 224 and L.device_status() == B.TIMEOUT
    L.set_tuning()
    L.reset_status()
    y = L.spmm_conv(x, 3, 3, 1, nhwc_out=True)
    torch.cuda.synchronize()
    assert L.device_status() == 0 and torch.equal(y, want)
    L.close()


@pytest.mark.parametrize("s_out,c,b,side,keep", [(168, 128, 28, 56, 0.5), (368, 64, 1, 224, 0.75)])
def test_results_stored_pixel_by_pixel_keep_two_accumulators(s_out, c, b, side, keep):
    """On one handle in turn: where TMA stores the results 256 pixels are the better tile, where they leave pixel by pixel 224, whatever was
    asked for before."""
    import torch
    import torch.nn.functional as F
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(s_out)
    L = B.HybridLayer(s_out, 9 * c, 2, 4, 64, 64, keep)
    L.build_mask(torch.rand(s_out, 9 * c, generator=g, device="cuda")).encode(torch.randn(s_out, 9 * c, generator=g, device="cuda").bfloat16())
    x = torch.randn(b, side, side, c, generator=g, device="cuda").bfloat16()
    # two orders of a sum of 9 c products differ by at most 2 * 9 c * 2^-23 * sum |w x|, their bf16 roundings by at most 2^-7 of the value
    mags = F.conv2d(x.float().abs().permute(0, 3, 1, 2), L.decode().float().abs().view(s_out, 3, 3, c).permute(0, 3, 1, 2), padding=1).permute(0, 2, 3, 1)
    first = None
    for pitch, tile in [(s_out, 256), (s_out + 4, 224), (s_out + 8, 256), (s_out + 1, 224), (s_out, 256)]:
        y = torch.full((b, side, side, pitch), 7.0, dtype=torch.bfloat16, device="cuda")
        L.spmm_conv(x, 3, 3, 1, y=y, nhwc_out=True)
        assert L.last_launch()["tile_cols"] == tile
        got = y[..., :s_out].float()
        assert bool((y[..., s_out:] == 7).all())
        if first is None:
            first = got
        assert bool(((got - first).abs() <= 2.0 ** -7 * first.abs() + 18 * c * 2.0 ** -23 * mags).all())
    L.close()
