"""A workspace sized for a batch serves a part of that batch, whatever row counts
the two launches would choose: the sizes below are ones where the part alone would
take fewer rows per lane, and so more hand-off rows, than the whole."""
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


@pytest.mark.parametrize("op, d, M, T, n, t, m", [
    ("align", 6, 754, 123, 1082, 113, 1082),
    ("score", 3, 3812, 142, 2795, 79, 2795),
    ("pairwise", 3, 0, 34, 1902, 27, 1858),
])
def test_workspace_of_the_whole_serves_a_part(wts, op, d, M, T, n, t, m):
    rng = np.random.default_rng(T)

    def batch(count, length):
        b = synth.pack([rng.normal(size=(length, d)).astype(np.float32) for _ in range(count)])
        return wts.Batch.from_numpy(b.data, b.offsets)

    code = {"align": _abi.OP_DTW_ALIGN, "score": _abi.OP_ANOMALY_SCORE, "pairwise": _abi.OP_PAIRWISE}[op]
    whole, part = batch(T, n), batch(t, m)
    room = wts.workspace_size(code, M, whole)
    assert room < wts.workspace_size(code, M, part)

    class Whole(wts.Workspace):
        def get(self, nbytes):
            return super().get(room)[:room]

    def call(ws):
        if op == "pairwise":
            return (wts.pairwise_dtw(part, None, ws),)
        B = torch.from_numpy(np.random.default_rng(1).normal(size=(M, d)).astype(np.float32)).cuda()
        return (wts.dtw_align if op == "align" else wts.anomaly_score)(B, part, None, ws)

    for x, y in zip(call(Whole()), call(wts.Workspace())):
        assert torch.equal(x, y)
