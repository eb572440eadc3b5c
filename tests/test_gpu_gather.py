"""Products on layouts TMA cannot address, on the tensor cores (spmm_gather.cu): edges of its tiles, parts of 32 and 64 rows,
every alignment of a row, walks split over 2, 4 and 8 CTAs, several tiles a CTA, against the oracle's product in 64 bits.

Tolerance: an fp32 accumulation of t products with one rounding (or truncation) per step is off by at most t * 2^-23 * sum |w x|;
the bf16 result (8 significant bits) adds at most 2^-8 of the value."""
import numpy as np
import pytest

import oracle
from helpers import bf16_dev, gpu_layer, oracle_layer, to_dev, y_to_f64
from paper_2311_14272_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [
    # rows, k, ncols, pitch, n, m, bm, bk, keep, offset of X's first element
    (160, 960, 49, 49, 2, 8, 32, 32, 0.5, 0),         # one column tile, walk split over 8
    (16, 420, 1, 1, 2, 4, 32, 32, 1.0, 1),            # one column, thirteen blocks and a bit
    (70, 600, 127, 127, 1, 8, 64, 96, 0.6, 3),        # 96-deep blocks, ragged rows, columns and k
    (130, 1000, 129, 140, 3, 4, 64, 64, 0.9, 4),      # one column beyond a tile, split; pitch a multiple of 8 bytes
    (256, 512, 3001, 3001, 1, 4, 64, 64, 0.5, 7),     # split over 2, odd pitch
    (300, 640, 2570, 2574, 4, 4, 128, 128, 0.4, 2),   # 128-deep blocks, as many weights as there can be
    (384, 256, 9004, 9004, 3, 8, 128, 32, 0.5, 4),    # more tiles than CTAs, 8-byte rows
    (64, 256, 20001, 20001, 8, 8, 32, 64, 0.5, 5),    # a thin layer (its image has two copies), odd rows
    (300, 700, 6076, 6076, 1, 4, 64, 64, 0.3, 0),
    (96, 160, 4100, 4100, 2, 4, 32, 128, 0.7, 6),
]


def make(rows, k, ncols, pitch, n, m, bm, bk, keep, off, favour=None):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(rows + ncols)
    w = wl.f32_to_bf16_bits(rng.standard_normal((rows, k)).astype(np.float32))
    s = rng.uniform(0.1, 2.0, (rows, k)).astype(np.float32)
    if favour is not None:
        favour(s)
    x = wl.f32_to_bf16_bits(rng.standard_normal((k, ncols)).astype(np.float32))
    L = gpu_layer(B, torch, w, s, n, m, bm, bk, keep)
    # what lies between the rows and around the matrix is not finite: it must not be used
    xbuf = torch.full((off + k * pitch,), float("nan"), dtype=torch.bfloat16, device="cuda")
    xv = torch.as_strided(xbuf, (k, ncols), (pitch, 1), off)
    xv.copy_(bf16_dev(x, torch))
    return torch, L, rng, w, s, x, xv


@pytest.mark.parametrize("rows,k,ncols,pitch,n,m,bm,bk,keep,off", CASES)
def test_product(rows, k, ncols, pitch, n, m, bm, bk, keep, off):
    torch, L, rng, w, s, x, xv = make(rows, k, ncols, pitch, n, m, bm, bk, keep, off)
    mk, vals, idx, wd, wb = oracle_layer(w, s, n, m, bm, bk, keep)
    bias = rng.standard_normal(rows).astype(np.float32)
    L.set_epilogue(to_dev(bias, torch), relu=True)
    ybuf = torch.full((rows * pitch + off + 1,), 5.0, dtype=torch.bfloat16, device="cuda")
    y = torch.as_strided(ybuf, (rows, ncols), (pitch, 1), off)
    L.spmm(xv, y=y)
    torch.cuda.synchronize()
    info = L.last_launch()
    assert info["path"] == 0 and info["tile_cols"] == 128 and L.device_status() == 0
    ref = oracle.bias_relu(oracle.spmm_fp64(wd, x), bias, True)
    x64 = np.abs(wl.bf16_bits_to_f32(x).astype(np.float64))
    terms = mk.kkeep * bk * n // m + 1
    bound = terms * 2.0 ** -23 * (np.abs(wd.astype(np.float64)) @ x64 + np.abs(bias)[:, None])
    bound = bound * (1 + 2.0 ** -8) + 2.0 ** -8 * np.abs(ref)
    assert np.all(np.abs(y_to_f64(y, torch) - ref) <= bound + 1e-30)
    outside = torch.ones_like(ybuf, dtype=torch.bool)
    torch.as_strided(outside, (rows, ncols), (pitch, 1), off).fill_(False)
    assert torch.all(ybuf[outside] == 5.0)
    L.close()


@pytest.mark.parametrize("rows,k,ncols,bm,bk", [(160, 960, 49, 32, 32), (256, 512, 9003, 64, 64)])
def test_values_that_are_not_finite_reach_only_the_rows_that_use_them(rows, k, ncols, bm, bk):
    """An infinity or a NaN under a pruned weight is not part of the sum, as in the kernel on the CUDA cores."""
    torch, L, rng, w, s, x, xv = make(rows, k, ncols, ncols, 2, 4, bm, bk, 0.5, 1)
    xv[3, ncols // 2] = float("inf")
    xv[k // 2, 0] = float("nan")
    xv[k - 1, ncols - 1] = -float("inf")
    y = L.spmm(xv)
    assert L.last_launch()["tile_cols"] == 128
    L.set_path(0)
    ref = L.spmm(xv)
    torch.cuda.synchronize()
    assert L.last_launch()["tile_cols"] == 0
    bad = ~torch.isfinite(ref)
    assert 0 < int(bad.sum()) < 3 * rows and torch.equal(bad, ~torch.isfinite(y))
    assert torch.equal(torch.isnan(ref), torch.isnan(y)) and torch.equal(ref[torch.isinf(ref)], y[torch.isinf(ref)])
    a, b = y[~bad].double(), ref[~bad].double()
    assert float((a - b).norm()) <= 2.0 ** -8 * float(b.norm())
    L.close()


def spoil(xv, where, torch):
    """Values that are not finite: one, a row and a column, one in a hundred, all."""
    k, ncols = xv.shape
    inf, nan = float("inf"), float("nan")
    if where == "one":
        xv[k // 2, ncols // 2] = inf
    elif where == "row and column":
        xv[k // 3, :] = -inf
        xv[:, ncols // 3] = nan
        xv[k - 1, ncols - 1] = inf
    elif where == "sprinkled":
        r = torch.rand(k, ncols, device="cuda", generator=torch.Generator(device="cuda").manual_seed(3))
        xv[r < 0.004] = inf
        xv[(r > 0.004) & (r < 0.007)] = -inf
        xv[(r > 0.007) & (r < 0.008)] = nan
    else:
        xv.fill_({"all NaN": nan, "all infinite": inf}[where])


SPOILT = [
    # rows, k, ncols, pitch, n, m, bm, bk, keep
    (160, 960, 49, 49, 2, 8, 32, 32, 0.5),            # walk split over 8
    (130, 1000, 131, 140, 3, 4, 64, 64, 0.9),         # split, ragged rows, 8-byte rows
    (256, 600, 6076, 6076, 1, 4, 64, 64, 0.25),
    (700, 300, 9001, 9001, 2, 4, 32, 128, 0.34),      # two tiles a CTA, odd rows
    (42, 70, 70001, 70004, 8, 8, 32, 96, 1.0),        # four tiles a CTA, k in the middle of a block
]


@pytest.mark.parametrize("rows,k,ncols,pitch,n,m,bm,bk,keep", SPOILT)
@pytest.mark.parametrize("where", ["one", "row and column", "sprinkled", "all NaN", "all infinite"])
@pytest.mark.parametrize("use_bias,relu,weights", [(False, False, False), (True, True, False), (True, False, True), (False, True, True)])
def test_values_that_are_not_finite(rows, k, ncols, pitch, n, m, bm, bk, keep, where, use_bias, relu, weights):
    """NaN and infinities of X, and of the weights and the bias, give what the kernel on the CUDA cores gives, and change no other result."""
    torch, L, rng, w, s, x, xv = make(rows, k, ncols, pitch, n, m, bm, bk, keep, 0)
    wd = bf16_dev(w, torch)
    if weights:
        wd[1, :] = 0.0                                          # a stored zero times an infinity is a NaN
        wd[2, ::3] = float("inf")
        wd[rows - 1, 1::5] = float("nan")
        L.encode(wd)
    bias = torch.randn(rows, device="cuda")
    bias[3] = -float("inf")
    L.set_epilogue(bias if use_bias else None, relu)
    spoil(xv, where, torch)
    y = L.spmm(xv)
    assert L.last_launch()["tile_cols"] == 128
    L.set_path(0)
    ref = L.spmm(xv)
    torch.cuda.synchronize()
    assert L.last_launch()["tile_cols"] == 0 and L.device_status() == 0
    assert torch.equal(torch.isnan(ref), torch.isnan(y))
    fin = torch.isfinite(ref)
    odd = ~fin & ~torch.isnan(ref)
    assert torch.equal(fin, torch.isfinite(y)) and torch.equal(ref[odd], y[odd])
    a, b = y[fin].double(), ref[fin].double()
    assert float((a - b).norm()) <= 2.0 ** -8 * float(b.norm())
    L.close()


@pytest.mark.parametrize("rows,k,ncols,n,m,bm,bk,keep", [(160, 960, 49, 2, 8, 32, 32, 0.5), (256, 2304, 6076, 1, 4, 64, 64, 0.25), (512, 4608, 588, 2, 4, 64, 64, 0.5)])
@pytest.mark.parametrize("where", ["one a column tile", "all NaN", "all infinite"])
def test_values_that_are_not_finite_cost_no_more_than_on_the_cuda_cores(rows, k, ncols, n, m, bm, bk, keep, where):
    torch, L, rng, w, s, x, xv = make(rows, k, ncols, ncols, n, m, bm, bk, keep, 0)
    if where == "one a column tile":
        xv[k // 2, 5::128] = float("inf")
    else:
        spoil(xv, where, torch)
    y = torch.empty(rows, ncols, dtype=torch.bfloat16, device="cuda")

    def time():
        times = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            for _ in range(20):
                L.spmm(xv, y=y)
            b.record()
            torch.cuda.synchronize()
            times.append(a.elapsed_time(b))
        return min(times)
    mine = time()
    L.set_path(0)
    assert mine <= 1.25 * time()
    L.close()


@pytest.mark.parametrize("ncols", [49, 9003])
def test_a_wait_that_runs_out_is_reported(ncols):
    torch, L, rng, w, s, x, xv = make(256, 640, ncols, ncols, 2, 4, 64, 64, 0.5, 0)
    want = L.spmm(xv)
    L.set_tuning(0, 2_000_000, 1)                      # the second fill gets no weight tile
    L.spmm(xv)
    assert L.device_status() == 6
    L.reset_status()
    L.set_tuning()
    y = L.spmm(xv)
    assert L.device_status() == 0 and torch.equal(y, want)
    L.close()


@pytest.mark.parametrize("ncols,limit", [(49, 1), (49, 20_000), (9003, 1), (9003, 20_000)])
def test_warps_that_give_up_at_different_times_leave_together(ncols, limit):
    """Short limits and a missing weight tile: the lanes of a warp find out one by one that there is nothing to wait for."""
    torch, L, rng, w, s, x, xv = make(256, 2048, ncols, ncols, 2, 4, 64, 64, 0.5, 0)
    want = L.spmm(xv)
    for fill in (0, 1, 2):                              # (a rank of the split walk has three)
        for _ in range(5):
            L.set_tuning(0, limit, fill)
            L.spmm(xv)
            assert L.device_status() == 6
            L.reset_status()
    L.set_tuning()
    y = L.spmm(xv)
    assert L.device_status() == 0 and torch.equal(y, want)
    L.close()


def test_products_of_two_threads_on_one_layer():
    """One layer, two host threads with a stream, an input and a row pitch each."""
    import threading
    torch, L, rng, w, s, x, xv = make(256, 640, 2049, 2049, 2, 4, 64, 64, 0.5, 0)
    xs = [xv, torch.randn(640, 1027, device="cuda").bfloat16()]
    wants = [L.spmm(v) for v in xs]
    gots = [torch.zeros_like(v) for v in wants]
    torch.cuda.synchronize()
    errors = []

    def work(i):
        with torch.cuda.stream(torch.cuda.Stream()):
            try:
                for _ in range(500):
                    L.spmm(xs[i], y=gots[i])
            except Exception as e:                       # noqa: BLE001 (reported by the test)
                errors.append(e)
    threads = [threading.Thread(target=work, args=(i,)) for i in range(2)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    assert errors == [] and L.device_status() == 0
    assert torch.equal(gots[0], wants[0]) and torch.equal(gots[1], wants[1])
    L.close()


def one_long_walk_in_nine(s):
    """Saliency of row tiles of 64 that all keep block 0, but for one of the 18, which keeps block 1."""
    s[:, :32] += 4.0
    s[576:640] = s[576:640, ::-1]


@pytest.mark.parametrize("rows,k,ncols,n,m,bm,bk,keep,favour", [
    (1034, 413, 2206, 3, 4, 64, 128, 0.4, None),        # a ring of two stages, walks of two or three blocks, two tiles a CTA
    (700, 300, 9001, 2, 4, 32, 128, 0.34, None),        # the same with the 2:4 image, walks of one or two blocks
    (1300, 800, 4999, 4, 4, 64, 96, 0.4, None),         # 96-deep blocks, walks of four to seven
    (1152, 64, 38401, 2, 4, 64, 32, 0.5, one_long_walk_in_nine),     # eight stages, walks of one block and every ninth of two
    (1152, 64, 38401, 4, 4, 64, 32, 0.5, one_long_walk_in_nine),
])
def test_several_tiles_with_walks_of_unlike_length(rows, k, ncols, n, m, bm, bk, keep, favour):
    """The two groups of X warps take every other block of all tiles of a CTA: neither may get ahead of the other by more than the ring.

    Reference: the kernel on the CUDA cores (checked against the oracle elsewhere).  Two orders of an fp32 sum of t products
    differ by at most 2 t * 2^-23 * sum |w x|, their bf16 roundings by at most 2^-7 of the value."""
    torch, L, rng, w, s, x, xv = make(rows, k, ncols, ncols, n, m, bm, bk, keep, 0, favour)
    mk, vals, idx, wd, wb = oracle_layer(w, s, n, m, bm, bk, keep)
    y = L.spmm(xv)
    info = L.last_launch()
    tiles = -(-rows // 128) * -(-ncols // 128)
    assert info["tile_cols"] == 128 and info["ctas"] < tiles
    walks = {len(set(mk.blk_col.reshape(-1, mk.kkeep)[i:i + 128 // bm].ravel())) for i in range(0, -(-rows // bm), 128 // bm)}
    assert len(walks) > 1
    L.set_path(0)
    ref = L.spmm(xv).double()
    torch.cuda.synchronize()
    assert L.last_launch()["tile_cols"] == 0 and L.device_status() == 0
    size = to_dev(np.abs(wd.astype(np.float64)), torch) @ xv.double().abs()
    terms = mk.kkeep * bk * n // m
    assert bool(((y.double() - ref).abs() <= 2.0 ** -7 * ref.abs() + 2 * terms * 2.0 ** -23 * size).all())
    L.close()


@pytest.mark.parametrize("rows,k,ncols,n,m,bm,bk,cuda_cores", [(49, 93, 7644, 1, 8, 128, 32, True), (191, 93, 2891, 2, 8, 32, 32, False)])
def test_many_results_of_few_weights(rows, k, ncols, n, m, bm, bk, cuda_cores):
    """One kept block of four or eight weights a row: which kernel takes it."""
    torch, L, rng, w, s, x, xv = make(rows, k, ncols, ncols, n, m, bm, bk, 0.34, 0)
    assert L.kkeep == 1
    y = L.spmm(xv)
    assert (L.last_launch()["tile_cols"] == 0) == cuda_cores
    L.set_path(0)
    ref = L.spmm(xv).double()
    torch.cuda.synchronize()
    assert float((y.double() - ref).norm()) <= 2.0 ** -8 * float(ref.norm())
    L.close()
