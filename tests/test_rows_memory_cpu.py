"""Rows per lane chosen by the launch's size stay within the workspace that a
caller can expect: at most 16 GiB more than the fixed rows take, and none more
past 64 GiB.  Host-side sizes only, no GPU."""
import ctypes

import numpy as np
import pytest

from paper_2404_12134_gb300 import _abi, build

GIB = 1 << 30


@pytest.fixture(scope="module")
def lib():
    build.build()
    return _abi.load()


def _size(lib, op, M, lens, d, **options):
    offs = np.concatenate([[0], np.cumsum(lens)]).astype(np.int64)
    b = _abi.wts_batch(16, 16, offs.ctypes.data, len(lens), d)     # (device pointers are not read)
    o = _abi.wts_options(**options)
    n = ctypes.c_size_t(0)
    assert lib.wts_workspace_size(op, M, ctypes.byref(b), ctypes.byref(o), ctypes.byref(n)) == 0
    return n.value


@pytest.mark.parametrize("op, T, M, d, cost_kind", [
    (_abi.OP_PAIRWISE, 200, 24500, 6, 1),      # the benchmark batch's medoid start under the l2 norm
    (_abi.OP_PAIRWISE, 1000, 4000, 6, 1),
    (_abi.OP_PAIRWISE, 400, 10000, 6, 1),
    (_abi.OP_PAIRWISE, 200, 24500, 2, 0),
    (_abi.OP_PAIRWISE, 250, 24500, 16, 0),
    (_abi.OP_DTW_ALIGN, 200, 60000, 6, 1),
    (_abi.OP_DBA_ITERATE, 60, 110000, 3, 1),
    (_abi.OP_ANOMALY_SCORE, 1000, 60000, 16, 0),
    (_abi.OP_SOFTDTW, 2, 8192, 1, 0),          # (M = 8,192 against cycles of millions: R alone is large)
])
def test_large_workspaces_do_not_grow(lib, op, T, M, d, cost_kind):
    lens = [3_000_000] * T if op == _abi.OP_SOFTDTW else [M] * T
    M = 0 if op == _abi.OP_PAIRWISE else M
    got = _size(lib, op, M, lens, d, cost_kind=cost_kind)
    if op == _abi.OP_SOFTDTW:
        # eight rows: R, the band rows (4 + 16 bytes a slot), and no more than the rest of the layout
        fixed = sum(8192 * (n + 31) * 4 + 31 * n * 20 for n in lens) + (64 << 20)
    else:
        fixed = _size(lib, op, M, lens, d, cost_kind=cost_kind, rows_per_thread=16 if d > 2 or cost_kind else 32)
    assert got <= max(fixed, min(fixed + 16 * GIB, 64 * GIB)), (got / GIB, fixed / GIB)


def test_small_batches_take_the_larger_workspace(lib):
    for op, T, M, d, cost_kind in ((_abi.OP_PAIRWISE, 16, 25000, 6, 1), (_abi.OP_ANOMALY_SCORE, 1, 1100, 1, 0),
                                   (_abi.OP_DTW_ALIGN, 24, 8191, 6, 1)):
        m = 0 if op == _abi.OP_PAIRWISE else M
        assert _size(lib, op, m, [M] * T, d, cost_kind=cost_kind) > _size(
            lib, op, m, [M] * T, d, cost_kind=cost_kind, rows_per_thread=16 if d > 2 or cost_kind else 32)


def test_pairwise_hand_off_slots_hold_the_cost_alone(lib):
    """Four bytes a slot for the pairwise matrix, at every row count (only the score
    counts path cells beside the cost)."""
    T, n, d = 12, 6000, 3
    bands = -(-n // 128)
    got = _size(lib, _abi.OP_PAIRWISE, 0, [n] * T, d)
    eight = _size(lib, _abi.OP_PAIRWISE, 0, [n] * T, d, rows_per_thread=8)
    pairs = T * (T - 1) // 2
    slots4, slots8 = pairs * (bands - 1) * n, pairs * (-(-n // 256) - 1) * n
    assert got > eight                         # four rows are the choice here
    assert abs((got - eight) - 4 * (slots4 - slots8)) <= 1024
