"""The CUDA-core product on layouts TMA cannot address (any row pitch, any 2-byte alignment), in each of its tile
forms, against the oracle's product in 64 bits.

Tolerance for fp32 results: sums of t products by fused multiply-adds, each rounded to fp32, are off by at most
t * 2^-24 * sum |w x| (first order); a bf16 result (8 significant bits) adds its own rounding, at most 2^-8 of the value."""
import numpy as np
import pytest

import oracle
from helpers import bf16_dev, gpu_layer, oracle_layer, to_dev, y_to_f64
from paper_2311_14272_b200 import workloads as wl

pytestmark = pytest.mark.gpu

CASES = [
    # rows, k, ncols, n, m, bm, bk, keep, offset of X's first element
    (160, 960, 49, 2, 8, 32, 32, 0.5, 0),        # one column tile, pitch odd
    (16, 33, 1, 2, 4, 32, 32, 1.0, 1),           # one column, one block and a bit
    (70, 200, 127, 1, 8, 64, 96, 0.6, 3),        # 3-bit offsets, 96-deep blocks, ragged rows and columns
    (256, 512, 3001, 1, 4, 64, 64, 0.5, 7),      # several column tiles, odd pitch
    (300, 640, 2570, 4, 4, 128, 128, 0.4, 2),    # as many weights per row and block as there can be; even pitch
    (384, 256, 9004, 3, 8, 128, 32, 0.5, 4),     # pitch a multiple of 8 bytes, widest form
    (64, 256, 20001, 8, 8, 32, 64, 0.5, 5),
]


@pytest.mark.parametrize("rows,k,ncols,n,m,bm,bk,keep,off", CASES)
@pytest.mark.parametrize("y_dtype", [0, 1])
def test_unaligned_product(rows, k, ncols, n, m, bm, bk, keep, off, y_dtype):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(rows + ncols)
    w = wl.f32_to_bf16_bits(rng.standard_normal((rows, k)).astype(np.float32))
    s = rng.uniform(0.1, 2.0, (rows, k)).astype(np.float32)
    x = wl.f32_to_bf16_bits(rng.standard_normal((k, ncols)).astype(np.float32))
    mk, vals, idx, wd, wb = oracle_layer(w, s, n, m, bm, bk, keep)
    L = gpu_layer(B, torch, w, s, n, m, bm, bk, keep)
    bias = rng.standard_normal(rows).astype(np.float32)
    L.set_epilogue(to_dev(bias, torch), relu=True)
    L.set_path(B.PATH_DIRECT)
    xbuf = torch.zeros(off + k * ncols, dtype=torch.bfloat16, device="cuda")
    xv = xbuf[off:].view(k, ncols)
    xv.copy_(bf16_dev(x, torch))
    ybuf = torch.full((rows * ncols + off + 1,), 5.0, dtype=torch.float32 if y_dtype else torch.bfloat16, device="cuda")
    y = ybuf[off:off + rows * ncols].view(rows, ncols)
    L.spmm(xv, y=y, y_dtype=y_dtype)
    torch.cuda.synchronize()
    assert L.last_launch()["path"] == B.PATH_DIRECT
    ref = oracle.bias_relu(oracle.spmm_fp64(wd, x), bias, True)
    x64 = np.abs(wl.bf16_bits_to_f32(x).astype(np.float64))
    terms = mk.kkeep * bk * n // m + 1
    bound = terms * 2.0 ** -24 * (np.abs(wd.astype(np.float64)) @ x64 + np.abs(bias)[:, None]) * 1.01
    if not y_dtype:
        bound = bound * (1 + 2.0 ** -8) + 2.0 ** -8 * np.abs(ref)
    assert np.all(np.abs(y_to_f64(y, torch) - ref) <= bound + 1e-30)
    assert torch.all(ybuf[:off] == 5.0) and torch.all(ybuf[off + rows * ncols:] == 5.0)
    L.close()


def test_products_of_falling_size_in_one_graph():
    """Two layers of one tile form, the one with more shared memory first, captured in one graph and replayed on new data."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(12)
    layers, xs, ys, refs = [], [], [], []
    for rows, k, n, m, bk, keep in ((128, 1024, 8, 8, 64, 1.0), (128, 512, 1, 8, 32, 0.25)):
        w = wl.f32_to_bf16_bits((rng.standard_normal((rows, k)) / 32).astype(np.float32))
        layers.append(gpu_layer(B, torch, w, np.abs(wl.bf16_bits_to_f32(w)) + 1e-3, n, m, 64, bk, keep))
        xs.append(torch.zeros(k, 49, dtype=torch.bfloat16, device="cuda"))
        layers[-1].set_path(B.PATH_DIRECT)
        ys.append(layers[-1].spmm(xs[-1]))
        assert layers[-1].last_launch()["path"] == 0 and layers[-1].last_launch()["tile_cols"] == 0
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        for L, x, y in zip(layers, xs, ys):
            L.spmm(x, y=y)
    for L, x in zip(layers, xs):
        x.copy_(torch.randn(x.shape, device="cuda"))
        refs.append(L.spmm(x))
    graph.replay()
    torch.cuda.synchronize()
    for L, y, ref in zip(layers, ys, refs):
        assert int((ref != 0).sum()) > 0 and torch.equal(y, ref)
        L.close()


def test_products_that_read_each_others_results():
    """A chain of products in a row, each reading what the one before wrote; the launches overlap."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(5)
    rows = 96
    layers = []
    for n, bk in ((2, 32), (3, 96), (1, 64)):                   # whole blocks, blocks in parts
        w = wl.f32_to_bf16_bits((rng.standard_normal((rows, rows)) / 4).astype(np.float32))
        layers.append(gpu_layer(B, torch, w, np.abs(wl.bf16_bits_to_f32(w)) + 1e-3, n, 4, 32, bk, 1.0))
        layers[-1].set_path(B.PATH_DIRECT)
    for ncols in (1, 49, 3001):
        xs = [torch.randn(rows, ncols, device="cuda").bfloat16() for _ in range(20)]
        wants, gots = [], []
        for x in xs:                                            # one at a time
            for L in layers:
                x = L.spmm(x)
                torch.cuda.synchronize()
            wants.append(x)
        bufs = [torch.zeros(rows, ncols, dtype=torch.bfloat16, device="cuda") for _ in layers]
        for x in xs:                                            # all in a row, through the same buffers
            for L, y in zip(layers, bufs):
                x = L.spmm(x, y=y)
            gots.append(x.clone())
        torch.cuda.synchronize()
        assert layers[0].last_launch()["tile_cols"] == 0
        for w, g in zip(wants, gots):
            assert torch.equal(w, g)
    for L in layers:
        L.close()
