"""The encode kernel and the batched pruning iteration against the oracle, bit for bit."""
import numpy as np
import pytest

import oracle
from helpers import assert_mask_and_encoding_equal, bf16_dev, check_tolerance, gpu_layer, oracle_layer, to_dev, y_to_f64
from paper_2311_14272_b200 import workloads as wl

pytestmark = pytest.mark.gpu

PATTERNS = [(n, 4) for n in range(1, 5)] + [(n, 8) for n in range(1, 9)]


@pytest.mark.parametrize("n,m", PATTERNS)
@pytest.mark.parametrize("rows,k,bm,bk,keep", [(130, 530, 32, 96, 0.5), (200, 256, 64, 128, 1.0), (257, 300, 128, 32, 0.4),
                                               (30, 200, 64, 64, 0.7)])
def test_encode_is_exact_and_the_image_multiplies(rows, k, bm, bk, keep, n, m):
    """Every N of both M: canonical format equal to the oracle's, and X = I through the image gives the weights back."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(rows * 100 + 10 * m + n)
    w = wl.f32_to_bf16_bits(rng.standard_normal((rows, k)).astype(np.float32))
    s = rng.uniform(0.1, 2.0, (rows, k)).astype(np.float32)
    mk, vals, idx, wd, wb = oracle_layer(w, s, n, m, bm, bk, keep)
    L = gpu_layer(B, torch, w, s, n, m, bm, bk, keep)
    assert_mask_and_encoding_equal(L, mk, vals, idx)
    cols = (k + 7) // 8 * 8
    eye = torch.eye(k, cols, dtype=torch.bfloat16, device="cuda")
    y = L.spmm(eye)
    assert L.last_launch()["path"] in (B.PATH_SPARSE, B.PATH_DENSE)
    got = y.view(torch.int16).cpu().numpy().view(np.uint16)
    assert np.array_equal(wl.bf16_bits_to_f32(got[:, :k]), wl.bf16_bits_to_f32(wb))
    L.close()


@pytest.mark.parametrize("n,m,bm,bk", [(2, 4, 64, 64), (3, 8, 32, 96), (1, 4, 128, 32)])
def test_batched_iteration_equals_the_layer_by_layer_calls(n, m, bm, bk):
    """Layers of odd sizes, gradients in bf16 and fp32 (also mixed, and as views with a row pitch that forbids 16-byte
    loads), one sample and several, more layers than one launch takes: the same S, scores, masks and encodings as the
    per-layer calls, and products through the encodings."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(bm + bk)
    shapes = [(1, 8), (33, 27), (130, 530), (64, 576), (257, 96)] + [(40 + i, 64 + 8 * i) for i in range(64)]
    weights, grads = [], []
    for i, (r, k) in enumerate(shapes):
        pad = 3 if i % 5 == 2 else 0
        w = torch.zeros((r, k + pad), dtype=torch.bfloat16, device="cuda")[:, :k]
        w.copy_(to_dev((rng.standard_normal((r, k)) * 0.1).astype(np.float32), torch))
        weights.append(w)
        gs = []
        for h in range(1 + i % 4):
            g = torch.zeros((r, k + pad), dtype=torch.float32 if (i + h) % 3 == 0 else torch.bfloat16, device="cuda")[:, :k]
            g.copy_(to_dev((rng.standard_normal((r, k)) * 1e-2).astype(np.float32), torch))
            gs.append(g)
        grads.append(gs)
    grads[3][0][5, 7] = float("nan")
    grads[3][1][6, 8] = float("inf")
    net = B.PruningNetwork(shapes, n, m, bm, bk)
    kk = net.step(weights, grads, 1.0 - 0.6 * n / m)
    torch.cuda.synchronize()
    ref, arr = [], []
    for (r, k), w, gs in zip(shapes, weights, grads):
        L = B.HybridLayer(r, k, n, m, bm, bk, 1.0)
        acc = torch.empty((r, k), dtype=torch.float32, device="cuda")
        s = torch.empty((r, k), dtype=torch.float32, device="cuda")
        for h, g in enumerate(gs):
            B.crisp_saliency_accumulate(g, 0 if g.dtype == torch.bfloat16 else 1, g.stride(0), r, k, acc, k, h == 0)
        B.crisp_saliency_finish_max(acc, k, w, w.stride(0), r, k, len(gs), s, k, L.workspace)
        L.build_mask_max_known(s)
        ref.append((L, s))
        arr.append(L.rank_layer(1))
    ra = B.make_rank_layers(arr)
    ws = torch.empty(B.crisp_global_rank_sizes(ra), dtype=torch.uint8, device="cuda")
    d_kk = torch.zeros(len(shapes), dtype=torch.int32, device="cuda")
    B.crisp_global_rank(ra, B.crisp_prune_fraction(1.0 - 0.6 * n / m, n, m), ws, d_kk)
    assert d_kk.cpu().tolist() == list(kk)
    for i, ((L, s), N, w, c) in enumerate(zip(ref, net.layers, weights, kk)):
        assert torch.equal(net.sal[i].view(torch.int32), s.view(torch.int32))
        words = 8 * L.nrt * L.nblk
        assert torch.equal(N.workspace[256:256 + words], L.workspace[256:256 + words])
        assert torch.equal(N.workspace[:4], L.workspace[:4])
        L.reselect(c).encode(w)
        for a, b in zip(L.export_mask() + L.export(), N.export_mask() + N.export()):
            assert np.array_equal(a, b)
        if 0 < i < 8 and c:
            x = torch.randn((w.shape[1], 72), device="cuda").to(torch.bfloat16)
            assert torch.equal(L.spmm(x), N.spmm(x)) and N.device_status() == 0
        L.close()
    net.close()


def test_more_samples_than_one_launch_takes():
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(3)
    w = wl.f32_to_bf16_bits((rng.standard_normal((32, 64)) * 0.1).astype(np.float32))
    g = (rng.standard_normal((641, 32, 64)) * 1e-2).astype(np.float32)
    net = B.PruningNetwork([(32, 64)], 2, 4, 32, 32)
    d_g = to_dev(g, torch)
    net.step([bf16_dev(w, torch)], [[d_g[i] for i in range(641)]], 0.5)
    assert np.array_equal(net.sal[0].cpu().numpy(), oracle.saliency_f32(g, w))
    net.close()


def test_prune_calls_refuse_bad_tables():
    import ctypes as C
    from paper_2311_14272_b200 import binding as B
    lib = B.load()
    arr = (B.PruneLayer * 2)()
    assert lib.crisp_prune_score(0, arr, None) == B.INVALID_ARG
    assert lib.crisp_prune_score(1, None, None) == B.INVALID_ARG
    assert lib.crisp_prune_score(1, arr, None) == B.BAD_SHAPE
    arr[0].desc = B.make_desc(32, 64, 2, 4, 32, 32, 1.0)
    arr[1].desc = B.make_desc(32, 64, 2, 8, 32, 32, 1.0)
    assert lib.crisp_prune_score(1, arr, None) == B.INVALID_ARG            # null pointers
    sz = (C.c_size_t * 2)()
    arr[0].kkeep = 3
    assert lib.crisp_prune_encode_sizes(1, arr, sz, sz) == B.INVALID_ARG   # two blocks per row tile
    m, h = (C.c_void_p * 2)(), (C.c_void_p * 2)()
    assert lib.crisp_prune_encode(2, arr, None, m, h) == B.INVALID_ARG and not any(m) and not any(h)
