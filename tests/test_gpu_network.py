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
    short = weights[0][:-1], weights[0][:, :-1]
    for bad in short:
        with pytest.raises(AssertionError):
            net.step([bad] + weights[1:], grads, 0.7)
    with pytest.raises(TypeError):
        B._network.table([], [])
    L = net.layers[0]
    with pytest.raises(B.CrispError):                     # nothing encoded yet
        L.decode()
    net.close()


@pytest.mark.parametrize("native", [True, False])
@pytest.mark.parametrize("in_turn", [False, True])
def test_gradients_of_another_kind_are_refused(native, in_turn, monkeypatch):
    """Before anything is launched that would read them."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    weights, grads = _inputs(torch, 8, 2)
    net = B.PruningNetwork(SHAPES, 2, 4, 32, 32)
    if not native:
        monkeypatch.setattr(B, "_network", False)
    g = grads[1][1]
    for bad in (g.half(), g.double(), g.t().contiguous().t(), g[:-1], g[:, :-1], g.cpu(), torch.cat([g, g], 1)[:, ::2]):
        given = [grads[0], [grads[1][0], bad], grads[2]]
        with pytest.raises(AssertionError):
            net.step(weights, (list(gs) for gs in given) if in_turn else given, 0.7)
    net.step(weights, grads, 0.7)
    net.close()


@pytest.mark.parametrize("native", [True, False])
def test_larger_gradients_and_those_of_convolutions(native, monkeypatch):
    """The layer's rows and columns of a larger matrix, and dense tensors of more dimensions, count as they lie."""
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    weights, grads = _inputs(torch, 9, 2)
    if not native:
        monkeypatch.setattr(B, "_network", False)
    forms = [lambda g: torch.nn.functional.pad(g, (0, 3, 0, 2)), lambda g: g.reshape(g.shape[0], -1, 2, 2),
             lambda g: g.reshape(g.shape[0], 2, 2, -1).permute(0, 3, 1, 2)]
    want = _run(B, torch, weights, grads)
    for form in forms:
        got = _run(B, torch, weights, [[form(g) for g in gs] for gs in grads])
        for a, b in zip(want, got):
            assert a[0] == b[0] and all(torch.equal(x, y) for x, y in zip(a[1], b[1]))
