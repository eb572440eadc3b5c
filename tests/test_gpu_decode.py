"""crisp_decode against the oracle, bit for bit: every N of both M, blocks 32 to 128 deep (96 does not divide the 256
columns a CTA writes), ragged edges, and output rows that are and are not aligned to 16 bytes."""
import numpy as np
import pytest

from helpers import gpu_layer, oracle_layer
from paper_2311_14272_b200 import workloads as wl

pytestmark = pytest.mark.gpu

PATTERNS = [(n, 4) for n in range(1, 5)] + [(n, 8) for n in range(1, 9)]
SHAPES = [(1, 8, 32, 32, 1.0, 0), (33, 250, 32, 64, 0.5, 0), (130, 520, 128, 96, 0.6, 3), (96, 1024, 64, 128, 0.4, 8)]


@pytest.mark.parametrize("n,m", PATTERNS)
@pytest.mark.parametrize("rows,k,bm,bk,keep,pad", SHAPES)
def test_decode_is_exact(rows, k, bm, bk, keep, pad, n, m):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(rows * 100 + 10 * m + n)
    w = wl.f32_to_bf16_bits(rng.standard_normal((rows, k)).astype(np.float32))
    s = rng.uniform(0.1, 2.0, (rows, k)).astype(np.float32)
    mk, vals, idx, wd, wb = oracle_layer(w, s, n, m, bm, bk, keep)
    L = gpu_layer(B, torch, w, s, n, m, bm, bk, keep)
    out = torch.full((rows, k + pad), 7.0, dtype=torch.bfloat16, device="cuda")
    B.crisp_decode(L.handle, out, k + pad)
    got = out.view(torch.int16).cpu().numpy().view(np.uint16)
    assert np.array_equal(got[:, :k], wb)
    assert torch.all(out[:, k:] == 7.0)                       # nothing written past k
    L.close()


def test_a_layer_knows_its_device():
    """Results of a layer made on "cuda" lie beside its buffers: the device is settled when the layer is made, not at each call."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    here = torch.device("cuda", torch.cuda.current_device())
    L = B.HybridLayer(64, 64, 2, 4, 32, 32, 1.0, device="cuda")
    assert L.device == here and L.mask_buf.device == here
    w = torch.randn(64, 64, device="cuda").bfloat16()
    L.build_mask(w.float().abs()).encode(w)
    assert L.decode().device == here and L.spmm(w).device == here
    L.close()
