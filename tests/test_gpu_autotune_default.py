"""The autotuner times what the default options run: where the choice of rows by the
launch's size is the fastest, it returns that choice."""
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


def _wavefront_ms(wts, call):
    call()
    best = float("inf")
    for _ in range(7):
        torch.cuda.synchronize()
        wts.profile_read("")
        wts.profile_enable(True)
        call()
        torch.cuda.synchronize()
        wts.profile_enable(False)
        best = min(best, wts.profile_read("wavefront")[0])
    return best


@pytest.mark.parametrize("T, N, d", [(4, 1100, 3), (16, 3000, 6)])
def test_tuned_is_not_slower_than_the_default(wts, T, N, d):
    """At these sizes four rows per lane are 1.2 to 1.5 times as fast as eight."""
    rng = np.random.default_rng(N)
    b = synth.pack([rng.normal(size=(N, d)).astype(np.float32) for _ in range(T)])
    gb = wts.Batch.from_numpy(b.data, b.offsets)
    B = torch.from_numpy(rng.normal(size=(N, d)).astype(np.float32)).cuda()
    for op, call in ((_abi.OP_ANOMALY_SCORE, wts.anomaly_score), (_abi.OP_DTW_ALIGN, wts.dtw_align)):
        opts, _ = wts.autotune(op, B, gb, wts.Workspace())
        ws = wts.Workspace()
        assert _wavefront_ms(wts, lambda: call(B, gb, opts, ws)) < 1.1 * _wavefront_ms(wts, lambda: call(B, gb, None, ws))
        for x, y in zip(call(B, gb, opts), call(B, gb)):
            assert torch.equal(x, y)
