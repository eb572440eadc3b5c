"""Block scores made from sums in a scale of their own, of 32 x 32 elements each: exact where the sum is shifted into the layer's scale, where it does not
stand and is counted again, and where nothing is left of it; for every form of the kernels, on S with any pitch and start."""
import numpy as np
import pytest

import oracle
from helpers import to_dev

pytestmark = pytest.mark.gpu

ROWS, K, BM, BK = 200, 700, 32, 32          # more than the kernel for small layers takes; edges in both directions


def _values(kind, rng):
    s = np.abs(rng.standard_normal((ROWS, K))).astype(np.float32) + 0.25
    e = np.zeros((ROWS, K), dtype=np.int64)
    if kind == "edge":                       # patches 15 to 19 binades below the largest: at 17 an element loses no bit, at 18 one
        e -= 15 + (np.arange(ROWS)[:, None] // 32 + np.arange(K)[None, :] // 32) % 5
        s *= 1 + np.float32(2.0 ** -23)
        e[5, 7] = 0
    elif kind == "mixed":                    # within a patch
        e -= rng.integers(0, 24, (ROWS, K))
    elif kind == "far":                      # 38 to 44 binades below, and zeros
        e -= 38 + (np.arange(ROWS)[:, None] // 32 + np.arange(K)[None, :] // 32) % 7
        s[64:96] = 0
        e[0, 0] = 0
    elif kind == "huge":                     # the scales at both ends of fp32
        e += 120 - 240 * (np.arange(K)[None, :] // 64 % 2)
    elif kind == "zeros":                    # kept zeros beside others
        s[rng.random((ROWS, K)) < 0.8] = 0
    return np.ldexp(s, e).astype(np.float32)


@pytest.mark.parametrize("n,m,mode", [(1, 4, 0), (2, 4, 0), (4, 4, 0), (1, 8, 0), (2, 8, 0), (3, 8, 0), (2, 4, 1)])
@pytest.mark.parametrize("kind", ["edge", "mixed", "far", "huge", "zeros"])
@pytest.mark.parametrize("pitch,start", [(704, 0), (708, 0), (701, 0), (712, 4), (712, 1)])
def test_scores(n, m, mode, kind, pitch, start):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    s = _values(kind, np.random.default_rng(n + 8 * m))
    mk = oracle.build_mask(s, n, m, BM, BK, 0.5, score_mode=mode)
    flat = torch.full((start + ROWS * pitch,), float("nan"), dtype=torch.float32, device="cuda")
    dev = torch.as_strided(flat, (ROWS, K), (pitch, 1), start)
    dev.copy_(to_dev(s, torch))
    L = B.HybridLayer(ROWS, K, n, m, BM, BK, 0.5, mode)
    L.workspace.fill_(255)
    L.build_mask(dev)
    got = L.workspace[256:256 + 8 * L.nrt * L.nblk].view(torch.int64).cpu().numpy().view(np.uint64)
    assert np.array_equal(got.reshape(L.nrt, L.nblk), np.asarray(mk.score, dtype=np.uint64).reshape(L.nrt, L.nblk))
    blk_col, nm_bits = L.export_mask()
    assert np.array_equal(blk_col, mk.blk_col) and np.array_equal(nm_bits, mk.nm_bits)
    L.close()


@pytest.mark.parametrize("n,m", [(2, 4), (1, 8), (3, 8)])
@pytest.mark.parametrize("spread", [0, 20])
def test_a_network_scores_as_its_layers_do(n, m, spread):
    """crisp_prune_score against build_mask of the saliency that it leaves, on layers with edges, gradients of both types."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(spread + n)
    shapes = [(200, 700), (33, 40), (96, 1032), (256, 36)]
    weights = [torch.randn(s, generator=g, device="cuda").bfloat16() for s in shapes]
    grads = [[torch.randn(s, generator=g, device="cuda") * torch.exp2(-spread * torch.rand(s, generator=g, device="cuda")) for _ in range(3)] for s in shapes]
    grads = [[gr.bfloat16() if i != 1 else gr for i, gr in enumerate(gs)] for gs in grads]
    net = B.PruningNetwork(shapes, n, m, 32, 32)
    net.step(weights, grads, 0.7)
    for L, sal in zip(net.layers, net.sal):
        one = B.HybridLayer(L.desc.rows, L.desc.k, n, m, 32, 32, 1.0).build_mask(sal)
        words = 8 * one.nrt * one.nblk
        assert torch.equal(one.workspace[256:256 + words], L.workspace[256:256 + words])
        assert torch.equal(one.workspace[:4], L.workspace[:4])
        mk = oracle.build_mask(sal.cpu().numpy(), n, m, 32, 32, 1.0)
        got = one.workspace[256:256 + words].view(torch.int64).cpu().numpy().view(np.uint64)
        assert np.array_equal(got, np.asarray(mk.score, dtype=np.uint64).ravel())
        one.close()
    net.close()
