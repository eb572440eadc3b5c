"""Convolutions of few output channels and short walks, whose weight tiles stay in shared memory, against the oracle's
convolution by definition: two to eight kept blocks, fewer rows than a tile has, ragged pixel tiles, both output layouts."""
import numpy as np
import pytest

import oracle
from helpers import bf16_dev, check_tolerance, gpu_layer, oracle_layer, to_dev, y_to_f64
from test_gpu_conv import conv_inputs

pytestmark = pytest.mark.gpu

CASES = [
    # s_out, k, pad, c, b, h, w, n, m, bm, keep          (enough pixels for 256-pixel tiles on half of the SMs)
    (64, 3, 1, 64, 11, 83, 84, 2, 4, 64, 0.4),            # four kept blocks, ragged in x and y
    (128, 3, 1, 64, 5, 64, 72, 1, 4, 128, 0.9),           # eight kept blocks: as many as stay
    (40, 1, 0, 128, 7, 56, 106, 2, 4, 64, 1.0),           # pointwise, two blocks, 40 rows
    (20, 3, 1, 64, 3, 115, 113, 3, 4, 32, 0.3),           # dense-tile image, 20 rows, odd sizes
    (96, 1, 0, 192, 6, 60, 64, 4, 8, 32, 0.67),           # three row tiles, union walk
]


@pytest.mark.parametrize("s_out,ks,pad,c,b,h,w,n,m,bm,keep", CASES)
@pytest.mark.parametrize("nhwc", [False, True])
@pytest.mark.parametrize("y_dtype", [0, 1])
def test_thin_convolution(s_out, ks, pad, c, b, h, w, n, m, bm, keep, nhwc, y_dtype):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    wt, sal, act = conv_inputs(s_out, ks, ks, c, b, h, w, seed=s_out + h)
    mk, vals, idx, wd, _ = oracle_layer(wt, sal, n, m, bm, 64, keep)
    bias = np.random.default_rng(s_out).standard_normal(s_out).astype(np.float32)
    ref = oracle.bias_relu(oracle.conv_fp64(wd, ks, ks, act, pad), bias, True)
    L = gpu_layer(B, torch, wt, sal, n, m, bm, 64, keep)
    L.set_epilogue(to_dev(bias, torch), relu=True)
    dt = torch.float32 if y_dtype else torch.bfloat16
    y = torch.full((b, h, w, s_out) if nhwc else (s_out, b * h * w), 7.0, dtype=dt, device="cuda")
    L.spmm_conv(bf16_dev(act, torch), ks, ks, pad, y=y, y_dtype=y_dtype, nhwc_out=nhwc)
    torch.cuda.synchronize()
    assert L.device_status() == 0
    assert L.last_launch()["tile_cols"] == 256 and L.last_launch()["epilogue_warps"] == 16     # the short-walk form
    assert L.last_resident_bytes() > 0                                                          # with its weight tiles kept
    got = y_to_f64(y, torch)
    check_tolerance(got.reshape(-1, s_out).T if nhwc else got, ref)
    L.close()


@pytest.mark.parametrize("s_out,ks,c,b,h,w,n,m,bm,keep,why", [
    (64, 1, 64, 8, 84, 84, 2, 4, 64, 1.0, "a walk of one block"),
    (64, 3, 64, 8, 84, 84, 2, 4, 64, 1.0, "a walk of nine blocks"),
    (160, 3, 64, 8, 84, 84, 2, 4, 64, 0.3, "two CTA tiles of rows"),
    (64, 3, 64, 1, 16, 16, 2, 4, 64, 0.4, "128-pixel tiles"),
])
def test_other_convolutions_load_their_weights_with_every_tile(s_out, ks, c, b, h, w, n, m, bm, keep, why):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    wt, sal, act = conv_inputs(s_out, ks, ks, c, b, h, w, seed=s_out + h)
    L = gpu_layer(B, torch, wt, sal, n, m, bm, 64, keep)
    L.spmm_conv(bf16_dev(act, torch), ks, ks, ks // 2)
    torch.cuda.synchronize()
    assert L.device_status() == 0 and L.last_resident_bytes() == 0
    L.close()


def test_bounded_wait_with_resident_weights():
    """The loads of every CTA's second fill are left out under a wait limit of about a millisecond: the kernel returns, the
    status says why, and the next product is right."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    s_out, ks, c, b, h, w, n, m, bm, keep = 64, 3, 64, 11, 83, 84, 2, 4, 64, 0.4
    wt, sal, act = conv_inputs(s_out, ks, ks, c, b, h, w, seed=3)
    _, _, _, wd, _ = oracle_layer(wt, sal, n, m, bm, 64, keep)
    L = gpu_layer(B, torch, wt, sal, n, m, bm, 64, keep)
    d_act = bf16_dev(act, torch)
    L.set_tuning(wait_limit_cycles=2_000_000, skip_fill=1)
    L.spmm_conv(d_act, ks, ks, 1)
    torch.cuda.synchronize()
    assert L.last_resident_bytes() > 0 and L.device_status() == B.TIMEOUT
    L.set_tuning()
    L.reset_status()
    y = L.spmm_conv(d_act, ks, ks, 1)
    torch.cuda.synchronize()
    assert L.last_resident_bytes() > 0 and L.device_status() == 0
    check_tolerance(y_to_f64(y, torch), oracle.conv_fp64(wd, ks, ks, act, 1))
    L.close()
