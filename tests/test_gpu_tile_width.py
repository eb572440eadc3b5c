"""Width of the column tiles of aligned products where dense tiles meet short walks: 256 columns with as many waves of
tiles as 192 take.  Reference: the kernel on the CUDA cores; two orders of a sum of at most 128 products, rounded to bf16."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,k,ncols,n,m,bm,bk,keep,width", [
    (55, 79, 39776, 3, 4, 64, 128, 1.0, 256), (267, 59, 17360, 3, 4, 64, 64, 0.71, 256), (749, 48, 26200, 4, 8, 64, 32, 0.63, 256),
    (200, 300, 11864, 3, 4, 64, 128, 0.6, 192),       # one wave of either width: the narrower
    (300, 640, 17360, 3, 4, 64, 64, 0.6, 192),        # longer walks take the width with the cheaper waves
])
def test_width(rows, k, ncols, n, m, bm, bk, keep, width):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(rows)
    w = torch.randn(rows, k, generator=g, device="cuda").bfloat16()
    L = B.HybridLayer(rows, k, n, m, bm, bk, keep)
    L.build_mask(w.float().abs()).encode(w)
    x = torch.randn(k, ncols, generator=g, device="cuda").bfloat16()
    y = L.spmm(x)
    assert L.last_launch()["tile_cols"] == width
    L.set_path(0)
    ref = L.spmm(x).double()
    torch.cuda.synchronize()
    assert L.device_status() == 0
    size = L.decode().double().abs() @ x.double().abs()
    assert bool(((y.double() - ref).abs() <= 2.0 ** -7 * ref.abs() + 2 * L.kkeep * bk * 2.0 ** -23 * size).all())
    L.close()
