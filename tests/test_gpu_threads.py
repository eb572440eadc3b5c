"""Host threads with layers, streams and buffers of their own: calls that run at the same time neither fail nor change each
other's results, although the layers need different amounts of shared memory of the same kernels."""
import threading

import pytest

pytestmark = pytest.mark.gpu


def run_together(torch, jobs, rounds):
    """Every job in a thread and stream of its own, `rounds` times each; the exceptions they ended with."""
    start, errors = threading.Barrier(len(jobs)), []

    def work(job):
        with torch.cuda.stream(torch.cuda.Stream()):
            start.wait()
            try:
                for _ in range(rounds):
                    job()
            except Exception as e:                       # noqa: BLE001 (reported by the test)
                errors.append(e)
    threads = [threading.Thread(target=work, args=(j,)) for j in jobs]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return errors


def make_layer(B, torch, rows, k, n, m, bm, bk, keep, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    w = torch.randn(rows, k, generator=g, device="cuda").bfloat16()
    L = B.HybridLayer(rows, k, n, m, bm, bk, keep)
    L.build_mask(w.float().abs()).encode(w)
    return L


# two layers of the same tile form (rows per warp, columns per lane, alignment): 88 and 75 KB of shared memory, or 75 and 55
@pytest.mark.parametrize("ncols", [49, 8 * 1024 + 2])
def test_direct_products_of_two_threads(ncols):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    layers = [make_layer(B, torch, 256, 2048, 8, 8, 64, 64, 1.0, 1), make_layer(B, torch, 256, 1024, 1, 8, 64, 32, 0.25, 2)]
    jobs, outs, refs = [], [], []
    for L in layers:
        x = torch.randn(L.desc.k, ncols, device="cuda").bfloat16()
        L.set_path(B.PATH_DIRECT)
        refs.append(L.spmm(x))
        assert L.last_launch()["path"] == 0 and L.last_launch()["tile_cols"] == 0        # the kernel on the CUDA cores
        y = torch.zeros_like(refs[-1])
        outs.append(y)
        jobs.append(lambda L=L, x=x, y=y: L.spmm(x, y=y))
    torch.cuda.synchronize()
    assert run_together(torch, jobs, 3000 if ncols < 1000 else 500) == []
    for y, ref in zip(outs, refs):
        assert torch.equal(y, ref)
    for L in layers:
        L.close()


def test_block_selections_of_two_threads():
    """Rows of more than 4090 blocks need more shared memory than a kernel has without asking."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    layers, refs = [], []
    for nblk, seed in ((4096, 1), (4091, 2)):
        L = make_layer(B, torch, 32, 32 * nblk, 2, 4, 32, 32, 1.0, seed)
        layers.append(L.reselect(nblk // 2))
        refs.append(L.export_mask())
    jobs = [lambda L=L: L.reselect(L.kkeep) for L in layers]
    assert run_together(torch, jobs, 3000) == []
    for L, (blk_col, nm_bits) in zip(layers, refs):
        got = L.export_mask()
        assert (got[0] == blk_col).all() and (got[1] == nm_bits).all()
        L.close()


def test_tensor_core_products_of_two_threads():
    """Two layers of the same kernel, planned anew at every call (the buffers alternate), one with a copy of its walk lists in
    shared memory beside the ring and one whose ring ends sooner."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    jobs, outs, refs, layers = [], [], [], []
    for (rows, k, keep, seed) in ((512, 1024, 0.5, 1), (640, 2048, 0.9, 2)):
        L = make_layer(B, torch, rows, k, 2, 4, 128, 64, keep, seed)
        x = torch.randn(k, 19200, device="cuda").bfloat16()
        refs.append(L.spmm(x))
        assert L.last_launch()["path"] == 2
        ys = [torch.zeros_like(refs[-1]), torch.zeros_like(refs[-1])]
        turn = [0]

        def job(L=L, x=x, ys=ys, turn=turn):
            turn[0] ^= 1
            L.spmm(x, y=ys[turn[0]])
        jobs.append(job)
        outs.append(ys)
        layers.append(L)
    torch.cuda.synchronize()
    assert run_together(torch, jobs, 500) == []
    for ys, ref, L in zip(outs, refs, layers):
        assert L.device_status() == 0
        assert torch.equal(ys[0], ref) and torch.equal(ys[1], ref)
        L.close()


def test_first_call_of_a_host_thread():
    """A product, or a convolution, as the first CUDA call of a thread, on buffers the layer has not seen: its tensor maps need
    a context that nothing has made current in that thread yet."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    L = make_layer(B, torch, 128, 64 * 9, 2, 4, 64, 64, 0.5, 5)
    x = torch.randn(64 * 9, 1024, device="cuda").bfloat16()
    act = torch.randn(2, 16, 16, 64, device="cuda").bfloat16()
    stream = torch.cuda.current_stream().cuda_stream
    want = [L.spmm(x), L.spmm_conv(act, 3, 3, 1)]
    got = [torch.zeros_like(w) for w in want]
    torch.cuda.synchronize()
    for call in (lambda: L.spmm(x, y=got[0], stream=stream), lambda: L.spmm_conv(act, 3, 3, 1, y=got[1], stream=stream)):
        errors = []

        def work():
            try:
                call()
            except Exception as e:                       # noqa: BLE001 (reported by the test)
                errors.append(e)
        t = threading.Thread(target=work)
        t.start()
        t.join()
        torch.cuda.synchronize()
        assert errors == []
    assert torch.equal(got[0], want[0]) and torch.equal(got[1], want[1])
    L.close()


@pytest.mark.parametrize("kind", ["shared taps", "one tap a load", "matrix", "matrix fp32", "all in turn"])
def test_one_layer_from_two_threads(kind):
    """Two threads with a stream, an input and a result each on one layer, whose plans for the last operands they take from each other."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    L = make_layer(B, torch, 128, 64 * 9, 2, 4, 64, 64, 0.5, 5)
    acts = [torch.randn(20, 28, 28, 64, device="cuda").bfloat16(), torch.randn(24, 14, 14, 64, device="cuda").bfloat16()]
    xs = [torch.randn(64 * 9, 4096, device="cuda").bfloat16(), torch.randn(64 * 9, 520, device="cuda").bfloat16()]
    calls = {
        "shared taps": lambda i, y: L.spmm_conv(acts[i], 3, 3, 1, y=y, nhwc_out=True),
        "one tap a load": lambda i, y: L.spmm_conv(acts[i], 3, 3, 1, y=y),
        "matrix": lambda i, y: L.spmm(xs[i], y=y),
        "matrix fp32": lambda i, y: L.spmm(xs[i], y=y, y_dtype=1),
    }
    names = list(calls)[:3] if kind == "all in turn" else [kind]
    wants = [[calls[n](i, None) for n in names] for i in range(2)]
    if kind == "shared taps":
        assert L.last_launch()["epilogue_warps"] == 16 and L.last_launch()["conv"] == 1
    gots = [[torch.zeros_like(w) for w in ws] for ws in wants]
    torch.cuda.synchronize()

    def job(i):
        for n, y in zip(names, gots[i]):
            calls[n](i, y)
    assert run_together(torch, [lambda: job(0), lambda: job(1)], 500) == []
    assert L.device_status() == 0
    for ws, gs in zip(wants, gots):
        for w, g in zip(ws, gs):
            assert torch.equal(w, g)
    L.close()
