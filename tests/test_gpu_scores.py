"""Block scores against the oracle's, exactly, for every form of the score kernel: n = 1 and 2 of both M (the groups'
largest values are selected), larger n and score mode 1 (mask bits or all elements); ties, zeros, infinities, NaN, denormals,
and a layer whose scale is no fp32 number."""
import numpy as np
import pytest

import oracle
from helpers import to_dev

pytestmark = pytest.mark.gpu


def _saliency(kind, rows, k, rng):
    s = rng.standard_normal((rows, k)).astype(np.float32)
    if kind == "ties":
        s = rng.integers(0, 3, (rows, k)).astype(np.float32)
    elif kind == "special":
        s[rng.random((rows, k)) < 0.1] = np.nan
        s[rng.random((rows, k)) < 0.05] = np.inf
        s[rng.random((rows, k)) < 0.05] = -np.inf
    elif kind == "denormal":
        s = (rng.integers(0, 1000, (rows, k)) * 1.4e-45).astype(np.float32)
    elif kind == "wide":
        s = (s * np.exp2(rng.integers(-60, 60, (rows, k)))).astype(np.float32)
    return s


@pytest.mark.parametrize("n,m,mode", [(1, 4, 0), (2, 4, 0), (1, 8, 0), (2, 8, 0), (3, 4, 0), (5, 8, 0), (2, 4, 1), (1, 8, 1)])
@pytest.mark.parametrize("kind", ["normal", "ties", "special", "denormal", "wide"])
@pytest.mark.parametrize("rows,k,bm,bk", [(70, 300, 32, 32), (130, 530, 64, 96), (128, 512, 128, 128)])
def test_scores_are_exact(n, m, mode, kind, rows, k, bm, bk):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    s = _saliency(kind, rows, k, np.random.default_rng(rows + 10 * n + m))
    mk = oracle.build_mask(s, n, m, bm, bk, 0.5, score_mode=mode)
    L = B.HybridLayer(rows, k, n, m, bm, bk, 0.5, mode)
    L.build_mask(to_dev(s, torch))
    got = L.workspace[256:256 + 8 * L.nrt * L.nblk].view(torch.int64).cpu().numpy().view(np.uint64)
    assert np.array_equal(got.reshape(L.nrt, L.nblk), np.asarray(mk.score, dtype=np.uint64).reshape(L.nrt, L.nblk))
    blk_col, nm_bits = L.export_mask()
    assert np.array_equal(blk_col, mk.blk_col) and np.array_equal(nm_bits, mk.nm_bits)
    L.close()
