"""PruningNetwork.step and HybridLayer.decode through csrc/network.cpp against the same in Python, for what the module takes itself and what it leaves to it."""
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(64, 576), (96, 40), (200, 300)]


def _inputs(torch, seed, samples):
    g = torch.Generator(device="cuda").manual_seed(seed)
    weights = [torch.randn(s, generator=g, device="cuda").bfloat16() for s in SHAPES]
    grads = [[torch.randn(s, generator=g, device="cuda").to(torch.bfloat16 if i % 2 else torch.float32) for i in range(samples)] for s in SHAPES]
    return weights, grads


def _run(B, torch, weights, grads, stream=None):
    net = B.PruningNetwork(SHAPES, 2, 4, 32, 32)
    out = []
    for kappa in (0.6, 0.8):                              # (the second replaces the first one's masks and handles)
        kept = net.step(weights, grads() if callable(grads) else grads, kappa, stream)
        if stream is not None:
            stream.synchronize()
        out.append((kept, [L.decode(stream) for L in net.layers], [L.desc.keep_ratio for L in net.layers], [L.kkeep for L in net.layers]))
    torch.cuda.synchronize()
    net.close()
    return out


class _Sub:
    """What only the Python code takes: an object with a tensor's methods."""

    def __init__(self, t):
        self._t = t

    def __getattr__(self, name):
        return getattr(self._t, name)


@pytest.mark.parametrize("form", ["lists", "tuples", "stacked", "iterable", "pitched", "parameter", "foreign", "stream"])
def test_same_as_in_python(form, monkeypatch):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    assert B._bind_network(), "csrc/network.cpp is not built"
    weights, grads = _inputs(torch, 5, 3)
    stream = None
    if form == "tuples":
        grads = tuple(tuple(gs) for gs in grads)
    elif form == "stacked":
        grads = [torch.stack([g.bfloat16() for g in gs]) for gs in grads]
    elif form == "iterable":
        held = grads
        grads = lambda: (list(gs) for gs in held)         # noqa: E731  (read anew by every step)
    elif form == "pitched":
        weights = [torch.nn.functional.pad(w, (0, 24))[:, :w.shape[1]] for w in weights]
        grads = [[torch.nn.functional.pad(g, (0, 7))[:, :g.shape[1]] for g in gs] for gs in grads]
    elif form == "parameter":
        weights = [torch.nn.Parameter(w) for w in weights]
    elif form == "foreign":
        grads = [[_Sub(g) for g in gs] for gs in grads]
    elif form == "stream":
        stream = torch.cuda.Stream()
        stream.wait_stream(torch.cuda.current_stream())
    native = _run(B, torch, weights, grads, stream)
    monkeypatch.setattr(B, "_network", False)
    plain = _run(B, torch, weights, grads, stream)
    for a, b in zip(native, plain):
        assert a[0] == b[0] and a[2] == b[2] and a[3] == b[3]
        assert all(torch.equal(x, y) for x, y in zip(a[1], b[1])) and any(bool((x != 0).any()) for x in a[1])


def test_wrong_weights_are_refused_as_before():
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    weights, grads = _inputs(torch, 6, 1)
    net = B.PruningNetwork(SHAPES, 2, 4, 32, 32)
    for bad in (weights[0].float(), weights[0].t().contiguous().t(), weights[0].cpu()):
        with pytest.raises(AssertionError):
            net.step([bad] + weights[1:], grads, 0.7)
    with pytest.raises(TypeError):
        B._network.table([], [])
    L = net.layers[0]
    with pytest.raises(B.CrispError):                     # nothing encoded yet
        L.decode()
    net.close()
