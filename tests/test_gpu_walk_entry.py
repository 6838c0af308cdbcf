"""The walk does not depend on what the range arrays hold on entry: neither its
result (stored codes and checkpointed groups, few and many segments) nor its time."""
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


def _inputs(wts, M, lens, d, integer=False):
    rng = np.random.default_rng(M + d)
    draw = (lambda n: rng.integers(-2, 3, size=(n, d))) if integer else (
        lambda n: np.cumsum(rng.normal(size=(n, d)), axis=0) * 0.2)
    b = synth.pack([draw(n).astype(np.float32) for n in lens])
    return torch.from_numpy(draw(M).astype(np.float32)).cuda(), wts.Batch.from_numpy(b.data, b.offsets)


# one segment, two, many; groups of one band and of several; rows that end a group
@pytest.mark.parametrize("M, lens, d, options", [
    (319, [1, 40, 700], 1, {}), (384, [2, 300], 3, {}), (385, [900, 1], 2, {}), (1093, [1000, 1200] * 3, 1, {}),
    (2500, [2600, 60, 2400], 6, {}), (2500, [2600, 60, 2400], 6, {"band": 0.2}),
    (2500, [2600, 60], 3, {"cost_kind": 1}),
    (1500, [1400, 1600, 30], 3, {"dir_mode": 1, "ckpt_bands": 1}), (2600, [2500, 900], 1, {"dir_mode": 1, "ckpt_bands": 2}),
    (3000, [2900, 3100], 6, {"dir_mode": 1, "ckpt_bands": 3, "band": 0.3}),
    (1024, [1000] * 1000, 1, {}),
])
def test_any_contents_give_the_one_walk(wts, M, lens, d, options):
    for integer in (False, True):
        B, gb = _inputs(wts, M, lens, d, integer)
        T = len(lens)
        # the reference: one band at a time, whose groups are no longer than a segment
        o1 = wts.options(**{**options, "dir_mode": 1, "ckpt_bands": 1, "rows_per_thread": 0 if options.get("band") or
                            options.get("cost_kind") else 8})
        want = wts.dtw_align(B, gb, o1, wts.Workspace())
        g = torch.Generator(device="cuda").manual_seed(M)
        for fill in ("junk", "zero", "exact"):
            jlo, jhi = (torch.zeros((T, M), dtype=torch.int32, device="cuda") for _ in range(2))
            if fill == "junk":
                for t in (jlo, jhi):
                    t.copy_(torch.randint(-5, max(lens) + 5, (T, M), generator=g, device="cuda"))
            elif fill == "exact":
                jlo.copy_(want[2])
                jhi.copy_(want[3])
            got = wts.dtw_align(B, gb, wts.options(**options), wts.Workspace(), jlo, jhi)
            for x, y in zip(got, want):
                assert torch.equal(x, y), (fill, integer)


@pytest.mark.parametrize("M, T, d, options", [(1093, 16, 1, {}), (8191, 24, 6, {}),
                                              (20000, 8, 1, {"dir_mode": 1, "ckpt_bands": 8})])
def test_time_does_not_depend_on_the_contents(wts, M, T, d, options):
    B, gb = _inputs(wts, M, [M - 13 * k for k in range(T)], d)
    o, ws = wts.options(**options), wts.Workspace()
    jlo, jhi = (torch.zeros((T, M), dtype=torch.int32, device="cuda") for _ in range(2))
    wts.dtw_align(B, gb, o, ws, jlo, jhi)
    exact = jlo.clone(), jhi.clone()

    def stage(a, b):
        best = float("inf")
        for _ in range(4):
            jlo.copy_(a)
            jhi.copy_(b)
            torch.cuda.synchronize()
            wts.profile_read("")
            wts.profile_enable(True)
            wts.dtw_align(B, gb, o, ws, jlo, jhi)
            torch.cuda.synchronize()
            wts.profile_enable(False)
            best = min(best, wts.profile_read("backtrack")[0])
        return best

    zeros = torch.zeros_like(jlo)
    assert stage(zeros, zeros) < 1.5 * stage(*exact)
