"""Products whose weight tiles and walk lists are read before the kernel in front of them has finished: never where that kernel is the one that
encodes them, in eager order, through handles that share buffers, across streams and in graphs, of products and of encodes.  The rule by itself is
tested in test_settled.py.  (The kernel for odd pitches, "odd" here, never reads early; its products settle the handle like the others.)"""
import ctypes as C

import pytest

pytestmark = pytest.mark.gpu


def _layer(B, torch, rows, k, n, m, bm, bk, g):
    L = B.HybridLayer(rows, k, n, m, bm, bk, 0.5)
    L.build_mask(torch.rand(rows, k, generator=g, device="cuda") + 0.1)
    return L


def _case(kind, torch, g):
    """-> rows, k, x, call(layer, x)"""
    if kind == "conv":
        x = torch.randn(4, 14, 14, 128, generator=g, device="cuda").bfloat16()
        return 128, 9 * 128, x, lambda L, x: L.spmm_conv(x, 3, 3, 1, nhwc_out=True)
    cols = {"tma": 512, "wide": 4096, "odd": 245}[kind]
    x = torch.randn(1024, cols, generator=g, device="cuda").bfloat16()
    return 256, 1024, x, lambda L, x: L.spmm(x)


@pytest.mark.parametrize("kind", ["tma", "wide", "odd", "conv"])
@pytest.mark.parametrize("n,m", [(2, 4), (3, 4)])
def test_every_product_takes_the_weights_encoded_last(kind, n, m):
    """A layer encoded over and over into the same buffers, two or three products after each, all of it queued behind other work."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(7)
    rows, k, x, call = _case(kind, torch, g)
    L = _layer(B, torch, rows, k, n, m, 64, 64, g)
    ws = [torch.randn(rows, k, generator=g, device="cuda").bfloat16() for _ in range(12)]
    refs = []
    for w in ws:
        L.encode(w)
        torch.cuda.synchronize()
        refs.append(call(L, x))
        torch.cuda.synchronize()
    assert not torch.equal(refs[0], refs[1])
    busy = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    outs = []
    for _ in range(12):
        busy.zero_()
    for i, w in enumerate(ws):
        L.encode(w)
        outs.append([call(L, x) for _ in range(1 + i % 3)])
    torch.cuda.synchronize()
    for ref, out in zip(refs, outs):
        assert all(torch.equal(ref, o) for o in out)
    L.close()


def test_a_handle_whose_buffers_another_encode_fills():
    """The first handle is kept, used, and used again right behind an encode of other weights into its buffers."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(9)
    rows, k, x, _ = _case("tma", torch, g)
    L = _layer(B, torch, rows, k, 2, 4, 64, 64, g)
    ws = [torch.randn(rows, k, generator=g, device="cuda").bfloat16() for _ in range(2)]
    L.encode(ws[0])
    refs, y = [], torch.empty(rows, x.shape[1], dtype=torch.bfloat16, device="cuda")
    busy = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    others = [B.crisp_encode(w, k, L.mask, L.canonical_buf, L.exec_buf) for w in ws]
    for h in others:
        B.crisp_destroy(h)
    for w in ws:
        h = B.crisp_encode(w, k, L.mask, L.canonical_buf, L.exec_buf)
        torch.cuda.synchronize()
        refs.append(L.spmm(x))
        torch.cuda.synchronize()
        B.crisp_destroy(h)
    for rep in range(20):
        busy.zero_()
        L.spmm(x, y=y)
        h = B.crisp_encode(ws[rep % 2], k, L.mask, L.canonical_buf, L.exec_buf)
        out = L.spmm(x)
        B.crisp_destroy(h)
        assert torch.equal(out, refs[rep % 2])
    L.close()


def test_streams_and_graphs():
    """A product in another stream than the last one, or one behind a product that was captured and has not run, follows an encode."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(11)
    rows, k, x, _ = _case("tma", torch, g)
    L = _layer(B, torch, rows, k, 2, 4, 64, 64, g)
    ws = [torch.randn(rows, k, generator=g, device="cuda").bfloat16() for _ in range(8)]
    refs = []
    for w in ws:
        L.encode(w)
        torch.cuda.synchronize()
        refs.append(L.spmm(x))
        torch.cuda.synchronize()
    a, b = torch.cuda.Stream(), torch.cuda.Stream()
    busy = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    y = torch.empty_like(refs[0])
    for i, (w, ref) in enumerate(zip(ws, refs)):
        with torch.cuda.stream(a):
            busy.zero_()
            L.encode(w)
            encoded = torch.cuda.Event()
            encoded.record()
        graph = torch.cuda.CUDAGraph()
        if i % 2:
            with torch.cuda.stream(b):
                b.wait_event(encoded)
                other = L.spmm(x)
        else:
            with torch.cuda.graph(graph, stream=b):
                L.spmm(x, y=y)
        with torch.cuda.stream(a):
            out = L.spmm(x)
        torch.cuda.synchronize()
        assert torch.equal(out, ref)
        if i % 2:
            assert torch.equal(other, ref)
        else:
            graph.replay()
            torch.cuda.synchronize()
            assert torch.equal(y, ref)
    L.close()


@pytest.mark.parametrize("kind", ["tma", "wide", "odd", "conv"])
@pytest.mark.parametrize("kept_handle", [False, True])
def test_replayed_encodes(kind, kept_handle):
    """A graph encodes again at every replay, into the buffers of the handle that was captured, or of one that was there before; products right in
    front of the replay and right behind it."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(13)
    rows, k, x, call = _case(kind, torch, g)
    L = _layer(B, torch, rows, k, 2, 4, 64, 64, g)
    ws = [torch.randn(rows, k, generator=g, device="cuda").bfloat16() for _ in range(6)]
    refs = []
    for w in ws:
        L.encode(w)
        torch.cuda.synchronize()
        refs.append(call(L, x))
        torch.cuda.synchronize()
    assert not torch.equal(refs[0], refs[1])
    w = ws[-1].clone()
    other = 0
    graph, stream = torch.cuda.CUDAGraph(), torch.cuda.Stream()
    with torch.cuda.graph(graph, stream=stream):
        if kept_handle:
            other = B.crisp_encode(w, k, L.mask, L.canonical_buf, L.exec_buf)
        else:
            L.encode(w)
    busy = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    torch.cuda.synchronize()
    outs = []
    for rep in range(3):
        for _ in range(4):
            busy.zero_()
        for i, new in enumerate(ws):
            w.copy_(new)
            graph.replay()
            outs.append((i, [call(L, x) for _ in range(1 + i % 3)]))
    torch.cuda.synchronize()
    for i, out in outs:
        assert all(torch.equal(refs[i], o) for o in out)
    del graph
    L.encode(ws[0])                                       # (and without the graph as before)
    assert all(torch.equal(refs[0], call(L, x)) for _ in range(3))
    B.crisp_destroy(other)
    L.close()


@pytest.mark.parametrize("kind", ["tma", "conv"])
def test_products_captured_in_a_stream_where_one_went_before(kind):
    """Such a product is captured as one that reads early; it is replayed behind an encode, first in its graph and behind another kernel."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(17)
    rows, k, x, call = _case(kind, torch, g)
    L = _layer(B, torch, rows, k, 2, 4, 64, 64, g)
    ws = [torch.randn(rows, k, generator=g, device="cuda").bfloat16() for _ in range(6)]
    refs = []
    for w in ws:
        L.encode(w)
        torch.cuda.synchronize()
        refs.append(call(L, x))
        torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    h = B.crisp_encode(ws[0], k, L.mask, L.canonical_buf, L.exec_buf)      # (later encodes fill the buffers of the handle whose products are captured)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.stream(stream):
        assert torch.equal(call(L, x), refs[0])
    with torch.cuda.graph(graph, stream=stream):
        first, second = call(L, x), call(L, x)
    busy = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
    for rep in range(3):
        for i, w in enumerate(ws):
            busy.zero_()
            B.crisp_destroy(h)
            h = B.crisp_encode(w, k, L.mask, L.canonical_buf, L.exec_buf)
            graph.replay()
            a, b = first.clone(), second.clone()
            eager = call(L, x)
            assert torch.equal(a, refs[i]) and torch.equal(b, refs[i]) and torch.equal(eager, refs[i])
    B.crisp_destroy(h)
    L.close()
