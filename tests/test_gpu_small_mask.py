"""Mask projections of small layers in one launch (mask_small_kernel), at the edges of what it takes: one to eight CTAs, more row tiles
than CTAs, ragged rows and columns, every block shape, score mode, no kept block, and the sizes beyond which the other kernels
run.  Bit-identical to the oracle, scores and maximum included."""
import numpy as np
import pytest

import oracle
from helpers import to_dev

pytestmark = pytest.mark.gpu

CASES = [
    # rows, k, n, m, bm, bk, keep, score mode, pitch
    (1, 1, 2, 4, 32, 32, 1.0, 0, 1),
    (25, 489, 2, 8, 32, 64, 0.96, 0, 489),            # one CTA, ragged, unaligned rows
    (70, 333, 3, 4, 32, 96, 0.5, 1, 340),             # three CTAs, all elements counted
    (256, 512, 2, 4, 32, 64, 0.5, 0, 512),            # eight CTAs with as many elements as they take
    (500, 100, 1, 4, 32, 128, 0.5, 0, 100),           # sixteen row tiles over eight CTAs
    (290, 60, 5, 8, 32, 32, 0.7, 0, 64),              # ten row tiles: two CTAs have two
    (128, 128, 4, 8, 128, 32, 0.0, 0, 128),           # no kept block
    (129, 100, 8, 8, 128, 32, 0.3, 0, 100),
    (512, 60, 2, 4, 32, 64, 1.0, 0, 60),              # two row tiles a CTA: the most
    (513, 60, 2, 4, 32, 64, 1.0, 0, 60),              # three: the kernels for any size
    (257, 512, 2, 4, 32, 64, 0.5, 0, 512),            # a row more than it takes: the kernels for any size
    (32, 544, 2, 4, 32, 32, 0.25, 0, 544),            # a block more than one CTA takes
]


@pytest.mark.parametrize("rows,k,n,m,bm,bk,keep,mode,pitch", CASES)
@pytest.mark.parametrize("kind", ["plain", "zeros and infinities", "all zero"])
def test_mask(rows, k, n, m, bm, bk, keep, mode, pitch, kind):
    import torch
    from paper_2311_14272_b200 import binding as B
    B.load()
    rng = np.random.default_rng(rows * 3 + k)
    s = rng.uniform(-2.0, 2.0, (rows, k)).astype(np.float32)
    if kind == "zeros and infinities":
        s[rng.random((rows, k)) < 0.3] = 0.0
        s[rng.random((rows, k)) < 0.02] = np.inf
        s[rng.random((rows, k)) < 0.02] = np.nan
        s[rng.random((rows, k)) < 0.05] *= np.float32(1e-30)
    elif kind == "all zero":
        s[:] = 0.0
    mk = oracle.build_mask(s, n, m, bm, bk, keep, score_mode=mode)
    L = B.HybridLayer(rows, k, n, m, bm, bk, keep, mode)
    sd = torch.full((rows, pitch), float("nan"), dtype=torch.float32, device="cuda")
    sd[:, :k] = to_dev(s, torch)
    L.mask_buf.fill_(255)
    L.workspace.fill_(255)
    for _ in range(2):                                   # (the second time on the first one's workspace)
        L.build_mask(sd[:, :k])
        blk_col, nm_bits = L.export_mask()
        assert np.array_equal(blk_col, mk.blk_col) and np.array_equal(nm_bits, mk.nm_bits)
    ws = L.workspace.cpu().numpy()
    score = ws[256:256 + 8 * L.nrt * L.nblk].view(np.uint64)
    canon = np.abs(np.where(np.isnan(s), 0, s))
    canon = np.minimum(canon, np.finfo(np.float32).max).astype(np.float32)
    assert ws[:4].view(np.float32)[0] == canon.max()
    assert np.array_equal(score.reshape(L.nrt, L.nblk), mk.score)
    # narrower on the scores left behind, and again with the maximum known
    if mk.kkeep > 1:
        L.reselect(mk.kkeep - 1)
        ref = oracle.build_mask(s, n, m, bm, bk, kkeep=mk.kkeep - 1, score_mode=mode)
        assert np.array_equal(L.export_mask()[0], ref.blk_col)
        L.build_mask_max_known(sd[:, :k])
        got = L.export_mask()
        assert np.array_equal(got[0], ref.blk_col) and np.array_equal(got[1], ref.nm_bits)
    L.close()
