"""What PruningNetwork hands to the library as an address and a pitch: which tensors hold a layer's rows, and that others are refused.  On the CPU, with
tensors that say they are on a GPU."""
import types

import pytest
import torch

from paper_2311_14272_b200 import binding as B

ROWS, K = 6, 20


class OnGpu(torch.Tensor):
    is_cuda = True


def _t(*shape, dtype=torch.float32):
    return torch.zeros(shape, dtype=dtype)


GOOD = {
    "matrix": _t(ROWS, K), "bf16": _t(ROWS, K, dtype=torch.bfloat16), "pitched": _t(ROWS, K + 4)[:, :K], "larger": _t(ROWS + 3, K + 5),
    "convolution": _t(ROWS, 5, 2, 2), "channels_last": _t(ROWS, 2, 2, 5).permute(0, 3, 1, 2), "pointwise": _t(ROWS, K, 1, 1),
    "one_in_between": _t(ROWS, 1, K), "fewer_rows_read": _t(2 * ROWS, K),
}
BAD = {
    "half": _t(ROWS, K, dtype=torch.float16), "double": _t(ROWS, K, dtype=torch.float64), "int": _t(ROWS, K, dtype=torch.int32),
    "transposed": _t(K, ROWS).t(), "few_rows": _t(ROWS - 1, K), "few_columns": _t(ROWS, K - 1), "every_other": _t(ROWS, 2 * K)[:, ::2],
    "broadcast": _t(ROWS, 1).expand(ROWS, K), "gaps": _t(ROWS, 5, 6)[:, :, :4], "none": _t(0, K), "scalar": torch.zeros(()),
    "stacked_halves": _t(2, ROWS // 2, K),
}


def _table(g):
    desc = B.make_desc(ROWS, K, 2, 4, 32, 32, 1.0)
    layer = types.SimpleNamespace(desc=desc, mask_buf=_t(1), workspace=_t(1))
    net = B.PruningNetwork.__new__(B.PruningNetwork)
    net.torch, net.sal = torch, [_t(ROWS, K)]
    arr = (B.PruneLayer * 1)()
    held = net._table(arr, [layer], [_t(ROWS, K, dtype=torch.bfloat16)], [[g]])
    return arr[0], held


@pytest.mark.parametrize("name", sorted(GOOD))
def test_taken(name):
    g = GOOD[name].as_subclass(OnGpu)
    entry, held = _table(g)
    assert (held[0][0], held[1][0], held[2][0]) == (g.data_ptr(), g.stride()[0], 0 if g.dtype is torch.bfloat16 else 1) and entry.samples == 1


@pytest.mark.parametrize("name", sorted(BAD))
def test_refused(name):
    with pytest.raises(AssertionError):
        _table(BAD[name].as_subclass(OnGpu))


def test_host_memory_is_refused():
    with pytest.raises(AssertionError):
        _table(GOOD["matrix"])


def test_one_column():
    assert B._holds_rows(_t(2, ROWS).t(), ROWS, 1) and B._holds_rows(_t(ROWS), ROWS, 1) and not B._holds_rows(_t(ROWS), ROWS + 1, 1)


def test_what_is_no_tensor_answers_for_itself():
    g = types.SimpleNamespace(data_ptr=lambda: 4096, stride=lambda: (K, 1), dtype=torch.float32)
    assert _table(g)[1][0][0] == 4096
