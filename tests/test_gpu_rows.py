"""Rows per lane chosen by the launch's size: four rows (the lean kernel) give
the same bits as an explicit row count, at the edges of its bands (128 rows), of
its blocks (8 columns) and of its lanes' ramp (31 steps), for every operation
that may run it; a workspace sized for the fixed rows is still accepted."""
import numpy as np
import pytest

from paper_2404_12134_gb300 import _abi, synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def wts():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2404_12134_gb300 import api, build
    build.build()
    return api


def _batch(wts, rng, lens, d, integer):
    draw = (lambda n: rng.integers(-3, 4, size=(n, d))) if integer else (lambda n: rng.normal(size=(n, d)))
    b = synth.pack([draw(n).astype(np.float32) for n in lens])
    return wts.Batch.from_numpy(b.data, b.offsets), draw


@pytest.mark.parametrize("d", [1, 4, 6, 9, 16])
@pytest.mark.parametrize("M", [1, 3, 4, 5, 127, 128, 129, 257, 700])
def test_few_rows_identical(wts, M, d):
    rng = np.random.default_rng(1000 * M + d)
    for integer in (False, True):
        gb, draw = _batch(wts, rng, [1, 2, 7, 8, 9, 30, 31, 32, 33, 39, 40, 41, 260], d, integer)
        B = torch.from_numpy(draw(M).astype(np.float32)).cuda()
        o = wts.options(rows_per_thread=16)
        for x, y in zip(wts.anomaly_score(B, gb), wts.anomaly_score(B, gb, o)):
            assert torch.equal(x, y)
        for x, y in zip(wts.dtw_align(B, gb, ws=wts.Workspace()), wts.dtw_align(B, gb, o, ws=wts.Workspace())):
            assert torch.equal(x, y)
        for x, y in zip(wts.dba_iterate(B, gb, ws=wts.Workspace()), wts.dba_iterate(B, gb, o, ws=wts.Workspace())):
            assert torch.equal(x, y)
        assert torch.equal(wts.pairwise_dtw(gb), wts.pairwise_dtw(gb, o))


@pytest.mark.parametrize("M", [1, 5, 127, 129, 300])
def test_few_rows_identical_l2(wts, M):
    rng = np.random.default_rng(M)
    for d, integer in ((1, True), (3, False), (9, False)):
        gb, draw = _batch(wts, rng, [1, 7, 8, 9, 31, 32, 33, 40, 200], d, integer)
        B = torch.from_numpy(draw(M).astype(np.float32)).cuda()
        a, o = wts.options(cost_kind=1), wts.options(cost_kind=1, rows_per_thread=16)
        for x, y in zip(wts.dtw_align(B, gb, a, wts.Workspace()), wts.dtw_align(B, gb, o, wts.Workspace())):
            assert torch.equal(x, y)
        assert torch.equal(wts.pairwise_dtw(gb, a), wts.pairwise_dtw(gb, o))


def test_overflowing_costs_identical(wts):
    """Finite samples whose squared differences overflow: every cost is +inf and
    ties decide, with few rows as with many."""
    rng = np.random.default_rng(5)
    gb, _ = _batch(wts, rng, [40, 70], 2, False)
    B = torch.full((150, 2), 3e38, device="cuda")
    o = wts.options(rows_per_thread=16)
    # the walk ends at the first column without reaching the start (|pi| = -1) and
    # leaves the ranges above as they were: zeros here
    def align(opt):
        ranges = [torch.zeros((2, 150), dtype=torch.int32, device="cuda") for _ in range(2)]
        return wts.dtw_align(B, gb, opt, wts.Workspace(), *ranges)

    for x, y in zip(align(None), align(o)):
        assert torch.equal(x, y)
    for x, y in zip(wts.anomaly_score(B, gb), wts.anomaly_score(B, gb, o)):
        assert torch.equal(x, y)


@pytest.mark.parametrize("cost", [0, 1])
@pytest.mark.parametrize("d", [1, 3, 8])
@pytest.mark.parametrize("M", [1, 3, 4, 127, 128, 129, 257, 600])
def test_soft_few_rows_identical(wts, M, d, cost):
    """Four rows (R kept, few pairs) against the checkpointed form, which holds
    eight: values and gradient bit for bit."""
    rng = np.random.default_rng(M + d)
    gb, draw = _batch(wts, rng, [1, 2, 8, 31, 32, 33, 64, 65, 300], d, False)
    B = torch.from_numpy(draw(M).astype(np.float32)).cuda()
    got = []
    for mode in (0, 1):
        o, ws = wts.options(cost_kind=cost, dir_mode=mode), wts.Workspace()
        v = wts.softdtw_forward(B, gb, 0.5, o, ws)
        got.append((v, wts.softdtw_backward(B, gb, 0.5, None, o, ws)))
        assert wts.read_status(ws.buf) == 0
    for x, y in zip(*got):
        assert torch.equal(x, y)


@pytest.mark.parametrize("op", ["score", "align"])
def test_workspace_of_the_fixed_rows_is_accepted(wts, op):
    rng = np.random.default_rng(6)
    gb, draw = _batch(wts, rng, [900, 1100], 6, False)
    B = torch.from_numpy(draw(1000).astype(np.float32)).cuda()
    code = _abi.OP_ANOMALY_SCORE if op == "score" else _abi.OP_DTW_ALIGN
    call = wts.anomaly_score if op == "score" else wts.dtw_align
    fixed = wts.workspace_size(code, 1000, gb, wts.options(rows_per_thread=16))
    assert fixed < wts.workspace_size(code, 1000, gb)

    class Small(wts.Workspace):
        def get(self, nbytes):
            return super().get(fixed)

    for x, y in zip(call(B, gb, None, Small()), call(B, gb, None, wts.Workspace())):
        assert torch.equal(x, y)
