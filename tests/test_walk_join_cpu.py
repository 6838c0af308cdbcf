"""A model, in plain Python, of the segmented backtrack: every segment walked at
once from a guessed cell above its top, then a pair's segments taken from the top
down and walked again where the path enters elsewhere, stopping at the first walk
(looked for only every few rows).  Against the one-walk backtrack on random code
matrices, whatever the range arrays hold on entry.  No GPU."""
import random

import numpy as np
import pytest

from test_walk_model_cpu import UP, LEFT, _move, one_walk


def _walk(code, i, j, lo, jlo, jhi, look, record_from):
    """From (i, j) down to row lo: (exit column or -1, failed, merged).  Rows above
    record_from are not recorded; look(i): whether the walk may merge on leaving row i."""
    while True:
        if i == 0 and j == 0:
            jlo[0] = 0
            return -1, False, False
        di, dj = _move(code, i, j)
        if (i == 0 and di) or (j == 0 and dj):
            return -1, True, False
        if di:
            merge = i - 1 >= lo and look(i) and jlo[i - 1] <= j - dj <= jhi[i - 1]
            if i <= record_from:
                jlo[i] = j
            if i - 1 <= record_from and i - 1 >= 0:
                jhi[i - 1] = j - dj
            if merge:
                return None, False, True
        i -= di
        j -= dj
        if i < lo:
            return j, False, False


def segmented(code, M, N, S, lead, groups, junk, rng):
    """Groups of rows from the top down (checkpointed codes), S rows a segment."""
    jlo, jhi = dict(junk), dict(junk)
    entry, bad = N - 1, False
    hi = M
    for rows in groups:
        lo = max(0, hi - rows)
        n = (hi - lo + S - 1) // S
        start, exit_, failed = [-1] * n, [-1] * n, [0] * n
        order = list(range(n))
        rng.shuffle(order)
        for k in order:
            top, bottom = min(hi, lo + (k + 1) * S) - 1, lo + k * S
            if not 0 <= entry < N:
                failed[k] = 1
                continue
            i = min(top + lead, hi - 1)
            j = entry if i == hi - 1 else i * entry // (hi - 1)
            ok = True
            while i > top:                      # above the segment: nothing recorded
                di, dj = _move(code, i, j)
                if j == 0 and dj:
                    ok = False
                    break
                i, j = i - di, j - dj
            if not ok:
                failed[k] = 1
                continue
            start[k], jhi[top] = j, j
            exit_[k], failed[k], _ = _walk(code, top, j, bottom, jlo, jhi, lambda i: False, top)
        above = exit_[n - 1]
        for k in range(n - 2, -1, -1):
            top, bottom = min(hi, lo + (k + 1) * S) - 1, lo + k * S
            if above == start[k]:
                above = exit_[k]
                continue
            if not 0 <= above < N:
                start[k], exit_[k], failed[k], above = above, -1, 1, -1
                continue
            may, old = not failed[k], exit_[k]
            at_top = may and jlo[top] <= above <= start[k]
            jhi[top] = start[k] = above
            if at_top:
                above = old
                continue
            look = (lambda i: rng.random() < 0.3) if may else (lambda i: False)
            e, f, merged = _walk(code, top, above, bottom, jlo, jhi, look, top)
            if merged:
                above = old
            else:
                exit_[k], failed[k], above = e, f, e
        bad |= any(failed) or any(start[k] != exit_[k + 1] for k in range(n - 1))
        entry = -1 if any(failed) or any(start[k] != exit_[k + 1] for k in range(n - 1)) else exit_[0]
        hi = lo
        if hi == 0:
            break
    plen = -1 if bad else sum(jhi[i] - jlo[i] + 1 for i in range(M))
    return plen, jlo, jhi


@pytest.mark.parametrize("grouped", [False, True])
def test_segments_joined_from_the_top_are_the_walk(grouped):
    rng = np.random.default_rng(17)
    order_rng = random.Random(5)
    for trial in range(500):
        M, N = int(rng.integers(1, 70)), int(rng.integers(1, 70))
        p = rng.dirichlet([1, 1, 1]) if trial % 2 else [0.8, 0.1, 0.1]
        code = rng.choice(3, size=(M, N), p=p).tolist()
        if trial % 13:
            for i in range(1, M):
                code[i][0] = UP
            for j in range(1, N):
                code[0][j] = LEFT
        S, lead = int(rng.integers(1, 20)), int(rng.integers(0, 25))
        junk = {i: int(rng.integers(-3, N + 3)) for i in range(M)}
        rows = int(rng.integers(1, 40)) if grouped else M
        want = one_walk(code, M, N)
        got = segmented(code, M, N, S, lead, [rows] * M, junk, order_rng)
        if want[0] < 0:
            assert got[0] == -1, trial
            continue
        assert got[0] == want[0], trial
        assert all(got[1][i] == want[1][i] and got[2][i] == want[2][i] for i in range(M)), trial
