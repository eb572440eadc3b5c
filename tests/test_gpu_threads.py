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
        refs.append(L.spmm(x))
        assert L.last_launch()["path"] == 0              # the direct product
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
