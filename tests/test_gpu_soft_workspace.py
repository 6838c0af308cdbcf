"""softdtw_backward told another workspace size than the forward: the rows per lane
then differ, R lies elsewhere, and the call says so instead of giving another
gradient."""
import ctypes

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


def test_backward_with_other_bytes_raises_the_status(wts):
    # ten bands of four rows take more hand-off rows than five of eight, and R the same
    M, d = 1280, 2
    rng = np.random.default_rng(3)
    b = synth.pack([rng.normal(size=(n, d)).astype(np.float32) for n in (900, 1300, 1000)])
    gb = wts.Batch.from_numpy(b.data, b.offsets)
    B = torch.from_numpy(rng.normal(size=(M, d)).astype(np.float32)).cuda()
    need = wts.workspace_size(_abi.OP_SOFTDTW, M, gb)
    lib = _abi.load()

    def backward(ws, nbytes):
        grad = torch.zeros_like(B)
        rc = lib.softdtw_backward(B.data_ptr(), M, ctypes.byref(gb.c()), 1.0, None, None, ws.buf.data_ptr(), nbytes,
                                  torch.cuda.current_stream().cuda_stream, grad.data_ptr())
        return rc, grad

    ws = wts.Workspace()
    wts.softdtw_forward(B, gb, 1.0, None, ws)
    rc, grad = backward(ws, need)
    assert rc == 0 and wts.read_status(ws.buf) == 0
    rc, other = backward(ws, need - 256)
    assert rc == 0
    if not torch.equal(grad, other):
        assert wts.read_status(ws.buf) == _abi.WTS_EINVAL
    # the next forward starts afresh, at either size
    for nbytes in (need - 256, need):
        v = torch.empty(3, device="cuda")
        assert lib.softdtw_forward(B.data_ptr(), M, ctypes.byref(gb.c()), 1.0, None, ws.buf.data_ptr(), nbytes,
                                   torch.cuda.current_stream().cuda_stream, v.data_ptr()) == 0
        rc, again = backward(ws, nbytes)
        assert rc == 0 and wts.read_status(ws.buf) == 0 and torch.equal(again, grad)
