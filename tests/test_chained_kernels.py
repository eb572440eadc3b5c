"""Kernels launched with programmatic dependent launch are alive while the kernels in front of them still write: checks on
the sources that such a kernel reads no data through the read-only path, which is defined only for data that nobody writes
during the kernel's life, and, on the GPU, that chains of them hand over what was written last."""
import glob
import os
import re

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2311_14272_b200", "csrc")
WAIT = re.compile(r"\b(?:chain_kernels|wait_for_prerequisites)\(\)")


def functions(text):
    """(header, name, body) of every function with a body at namespace level."""
    text = re.sub(r"//[^\n]*|/\*.*?\*/|__launch_bounds__\([^()]*\)", "", text, flags=re.S)
    for m in re.finditer(r"((?:__global__|__device__)[^;{}]*?(\w+)\s*\([^;{}]*\))\s*\{", text):
        depth, at = 1, m.end()
        while depth:
            depth += {"{": 1, "}": -1}.get(text[at], 0)
            at += 1
        yield m.group(1), m.group(2), text[m.end():at - 1]


def chained_kernels():
    out = {}
    for path in sorted(glob.glob(os.path.join(CSRC, "*.cu"))):
        text = open(path).read() + "".join(open(p).read() for p in sorted(glob.glob(os.path.join(CSRC, "*.cuh"))))
        fns = list(functions(text))
        for header, name, body in fns:
            if "__global__" not in header or not WAIT.search(body):
                continue
            # with the device functions it calls, and theirs
            reached, todo = {}, [body]
            while todo:
                b = todo.pop()
                for h, n, inner in fns:
                    if n not in reached and "__global__" not in h and re.search(r"\b%s\b\s*[<(]" % n, b):
                        reached[n] = h + "{" + inner + "}"
                        todo.append(inner)
            out[name] = (header, body, reached)
    return out


def test_the_chained_kernels_are_found():
    assert {"encode_kernel", "decode_kernel", "block_score_kernel", "block_select_kernel", "clear_scores_kernel",
            "saliency_bits_kernel", "spmm_tc_kernel"} <= set(chained_kernels())


@pytest.mark.parametrize("name", sorted(chained_kernels()))
def test_chained_kernel_has_no_read_only_loads(name):
    header, body, reached = chained_kernels()[name]
    for where, text in [(name, header + body)] + sorted(reached.items()):
        assert "__ldg" not in text and "ld.global.nc" not in text, where
        assert not re.search(r"\bconst\b[^,;()=]*__restrict__", text), where


@pytest.mark.parametrize("name", sorted(chained_kernels()))
def test_no_exit_of_a_chained_kernel_before_its_wait(name):
    """The kernel behind it waits for this one alone: that it also comes after the one in front of this one holds only if
    every thread of this one waited."""
    _, body, _ = chained_kernels()[name]
    last = [w.start() for w in WAIT.finditer(body)][-1]
    for r in re.finditer(r"\breturn\b", body[:last]):
        assert WAIT.search(body, body.rfind("{", 0, r.start()), r.start()), body[:r.end()][-200:]


@pytest.mark.gpu
@pytest.mark.parametrize("n,m,bm,bk", [(2, 4, 128, 64), (4, 8, 32, 32), (3, 4, 64, 96)])
def test_chain_of_encode_and_decode_hands_over_the_newest_data(n, m, bm, bk):
    """mask, encode and decode of one layer's buffers over and over, with new weights each time and no wait between."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rows, k, rounds = 640, 1152, 24
    g = torch.Generator(device="cuda").manual_seed(n * 100 + bm)
    ws = [torch.randn(rows, k, generator=g, device="cuda").bfloat16() for _ in range(rounds)]
    L = B.HybridLayer(rows, k, n, m, bm, bk, 0.5)
    outs, again = [], []
    for w in ws:
        L.build_mask(w.float().abs()).encode(w)
        outs.append(L.decode())
        L.encode(outs[-1])                        # the weights of this encode are what decode just wrote
        again.append(L.decode())
    # the same, each call finished before the next
    for w, out, out2 in zip(ws, outs, again):
        sal = w.float().abs()
        torch.cuda.synchronize()
        L.build_mask(sal)
        torch.cuda.synchronize()
        L.encode(w)
        torch.cuda.synchronize()
        ref = L.decode()
        torch.cuda.synchronize()
        assert int((ref != 0).sum()) > 0
        assert torch.equal(ref.view(torch.int16), out.view(torch.int16))
        assert torch.equal(ref.view(torch.int16), out2.view(torch.int16))
    L.close()


@pytest.mark.gpu
@pytest.mark.parametrize("graph", [False, True])
@pytest.mark.parametrize("rows,k,n,m,bm,bk", [(64, 256, 2, 4, 32, 32), (512, 1024, 3, 8, 64, 64), (2048, 2048, 2, 4, 128, 64)])
def test_encode_and_decode_of_one_mask_with_new_weights_each_time(rows, k, n, m, bm, bk, graph):
    """One buffer is written by every encode and read by the decode behind it, which is still there when the next encode's
    launch begins: queued behind other work, or captured in one graph, every decode gives its own encode's weights."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    g = torch.Generator(device="cuda").manual_seed(rows + n)
    ws = [torch.randn(rows, k, generator=g, device="cuda").bfloat16() for _ in range(16)]
    L = B.HybridLayer(rows, k, n, m, bm, bk, 0.5)
    L.build_mask(torch.rand(rows, k, generator=g, device="cuda") + 0.1)
    refs = []
    for w in ws:
        L.encode(w)
        torch.cuda.synchronize()
        refs.append(L.decode())
        torch.cuda.synchronize()
    kept = refs[0] != 0
    assert 0 < int(kept.sum()) < kept.numel()
    for w, ref in zip(ws, refs):
        assert torch.equal(ref, torch.where(kept, w, torch.zeros_like(w)))
    outs = []

    def chain():
        for w in ws:
            L.encode(w)
            outs.append(L.decode())

    if graph:
        captured = torch.cuda.CUDAGraph()
        with torch.cuda.graph(captured):
            chain()
        for _ in range(3):
            captured.replay()
    else:
        busy = torch.empty(1 << 28, dtype=torch.uint8, device="cuda")
        for _ in range(3):
            outs.clear()
            for _ in range(20):                       # the chain is queued before the first of it runs
                busy.zero_()
            chain()
    torch.cuda.synchronize()
    for out, ref in zip(outs, refs):
        assert torch.equal(out, ref)
    L.close()
