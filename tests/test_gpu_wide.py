"""Seven to sixteen channels with eight and sixteen rows per lane: the same bits as
four rows (another kernel), at the edges of lanes, bands and chunks, in every form;
and sixteen channels within reach of twelve in time (their prototype rows spill,
and what holds the spills must not be taken)."""
import numpy as np
import pytest

from paper_2404_12134_gb300 import synth

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
    draw = (lambda n: rng.integers(-2, 3, size=(n, d))) if integer else (lambda n: rng.normal(size=(n, d)))
    b = synth.pack([draw(n).astype(np.float32) for n in lens])
    return wts.Batch.from_numpy(b.data, b.offsets), draw


@pytest.mark.parametrize("d", [7, 8, 10, 12, 13, 16])
@pytest.mark.parametrize("M", [1, 7, 9, 255, 256, 257, 511, 513, 800])
def test_rows_identical(wts, M, d):
    rng = np.random.default_rng(100 * M + d)
    for integer in (False, True):
        gb, draw = _batch(wts, rng, [1, 30, 31, 32, 33, 63, 64, 65, 127, 128, 129, 161, 330], d, integer)
        B = torch.from_numpy(draw(M).astype(np.float32)).cuda()
        for rows in (8, 16):
            o = wts.options(rows_per_thread=rows)
            for call in (wts.anomaly_score, wts.dtw_align, wts.dba_iterate):
                for x, y in zip(call(B, gb, o, wts.Workspace()), call(B, gb, None, wts.Workspace())):
                    assert torch.equal(x, y)
            assert torch.equal(wts.pairwise_dtw(gb, o), wts.pairwise_dtw(gb))
            for x, y in zip(wts.subdtw_align(B, gb, o), wts.subdtw_align(B, gb, wts.options(rows_per_thread=4))):
                assert torch.equal(x, y)
        l2, l2r = wts.options(cost_kind=1), wts.options(cost_kind=1, rows_per_thread=16)
        for x, y in zip(wts.dtw_align(B, gb, l2, wts.Workspace()), wts.dtw_align(B, gb, l2r, wts.Workspace())):
            assert torch.equal(x, y)
        # checkpointed groups, and a band that leaves no cell out
        for o in (wts.options(dir_mode=1, ckpt_bands=1, rows_per_thread=8), wts.options(dir_mode=1, ckpt_bands=1),
                  wts.options(band=1.0)):
            for x, y in zip(wts.dtw_align(B, gb, o, wts.Workspace()), wts.dtw_align(B, gb, None, wts.Workspace())):
                assert torch.equal(x, y)


def test_sixteen_channels_within_reach_of_twelve(wts):
    """Wavefront time of a pair, 16 rows per lane, 16 against 12 channels: about 2.1 times
    (3.9 with 170 KB of shared memory for the blocks of an SM, which leaves 60 KB of L1)."""
    rng = np.random.default_rng(1)

    def per_pair(d, T):
        gb, draw = _batch(wts, rng, [5000] * T, d, False)
        B = torch.from_numpy(draw(5000).astype(np.float32)).cuda()
        o, ws = wts.options(rows_per_thread=16), wts.Workspace()
        best = float("inf")
        for _ in range(4):
            wts.profile_read("")
            wts.profile_enable(True)
            wts.anomaly_score(B, gb, o, ws)
            torch.cuda.synchronize()
            wts.profile_enable(False)
            best = min(best, wts.profile_read("wavefront")[0])
        return best / T

    assert per_pair(16, 120) < 2.8 * per_pair(12, 240)
