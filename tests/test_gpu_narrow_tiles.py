"""Products with at most one tile of 64 columns for every SM: the line itself, ragged edges in all three sizes, both images, both result types."""
import numpy as np
import pytest

from helpers import to_dev

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(2, 4), (3, 4), (1, 8)])
@pytest.mark.parametrize("f32", [False, True])
@pytest.mark.parametrize("rows,k,tiles", [(40, 70, 1), (128, 64, 2), (129, 520, 9), (300, 1100, 73), (4096, 96, 4), (96, 200, "line"), (256, 300, "beyond")])
def test_result_and_width(n, m, f32, rows, k, tiles):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    sms, nst = torch.cuda.get_device_properties(0).multi_processor_count, -(-rows // 128)
    boxes = {"line": sms // nst, "beyond": sms // nst + 1}.get(tiles, tiles)
    ncols = 64 * boxes - 24 if boxes > 1 else 40                  # (a multiple of 8; the last tile is not full)
    g = torch.Generator(device="cuda").manual_seed(rows + k)
    w = torch.randn(rows, k, generator=g, device="cuda").bfloat16()
    x = torch.randn(k, ncols, generator=g, device="cuda").bfloat16()
    bias = torch.randn(rows, generator=g, device="cuda")
    L = B.HybridLayer(rows, k, n, m, 64, 64, 0.6 if k > 64 else 1.0)
    L.build_mask(w.float().abs()).encode(w)
    L.set_epilogue(bias, True)
    guard = torch.full((rows + 1, ncols), 7.0, dtype=torch.float32 if f32 else torch.bfloat16, device="cuda")
    y = L.spmm(x, y=guard[:rows], y_dtype=1 if f32 else 0)
    ref = (L.decode().double() @ x.double() + bias.double()[:, None]).clamp_(min=0)
    assert bool((guard[rows] == 7).all())
    # fp32: sums of at most 1100 terms; bf16 results: their rounding, half a unit of 2^-8
    bound = (2.0 ** -8 * 1.01 * ref if not f32 else 0) + 1100 * 2.0 ** -24 * (w.double().abs() @ x.double().abs() + 1)
    assert bool(((y.double() - ref).abs() <= bound).all())
    width = L.last_launch()["tile_cols"]
    assert width == 64 if nst * boxes <= sms else width > 64
    L.close()
