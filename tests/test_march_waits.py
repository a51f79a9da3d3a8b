"""The rows' waits of a 2D pass (await_rows, await_slot and the block barrier of
csrc/march.cuh) as a model under random schedules: sixteen warps take the rows of
a chunk in turn, a parity wait answers as an mbarrier's does, and +-y groups live
in one place per row slot and level.  For passes of two, three and four levels
and chunks of every length around the sixteen rows in flight: each wait is over
exactly when its phase is, each group read is the neighbour's, and every row
ends."""
import random

import pytest

ROWS = 16


def _pass(rows, n, seed, slot_wait=True, barrier=True):
    rng = random.Random(seed)
    done = [[0] * n for _ in range(ROWS)]     # completed phases per slot and level
    group = {}                                # (slot, level): the row whose groups lie there
    arrived = set()

    def waits(i, w, l, last):
        above, below = (w - 1) % ROWS, (w + 1) % ROWS
        if l == 0:
            if n == 2 and i >= ROWS and slot_wait:
                if i != ROWS:
                    yield above, 1, i - ROWS - 1
                yield below, 1, i - ROWS + 1
            return
        if i > 0:
            yield above, l - 1, i - 1
        if i != last:
            yield below, l - 1, i + 1
        elif i >= ROWS - 1:
            yield below, n - 1, i - (ROWS - 1)

    def warp(w):
        i = w
        if i >= rows:
            arrived.add(w)
        while i < rows:
            for l in range(n):
                if l == 1 and i < ROWS:
                    arrived.add(w)
                    while barrier and len(arrived) < ROWS:
                        yield
                for slot, lev, row in waits(i, w, l, rows - 1):
                    while done[slot][lev] % 2 == row // ROWS % 2:
                        yield
                    assert slot == row % ROWS and done[slot][lev] == row // ROWS + 1
                yield
                for row in (i - 1, i + 1):
                    if l > 0 and 0 <= row < rows:
                        for _ in range(2):    # a read takes its time
                            assert group[row % ROWS, l - 1] == row
                            yield
                if l < n - 1:
                    group[w, l] = i
                    yield
                done[w][l] += 1
                yield
            i += ROWS

    live = {w: warp(w) for w in range(ROWS)}
    for _ in range(4000):                     # stretches in which some warps are far faster than others
        speed = [rng.choice((1, 1, 20, 200)) for _ in range(ROWS)]
        for _ in range(rng.choice((5, 50, 500))):
            if not live:
                return
            warps = list(live)
            w = rng.choices(warps, [speed[v] for v in warps])[0]
            if next(live[w], "ended") == "ended":
                del live[w]
    raise AssertionError("rows that never end")


@pytest.mark.parametrize("n", [2, 3, 4])
def test_waits_hold_under_random_schedules(n):
    for rows in (1, 2, 3, 15, 16, 17, 18, 19, 31, 32, 33, 34, 49, 50, 65, 100):
        for seed in range(4):
            _pass(rows, n, seed)


@pytest.mark.parametrize("n,left_out", [(2, "slot_wait"), (2, "barrier"), (4, "barrier")])
def test_the_model_sees_a_wait_left_out(n, left_out):
    with pytest.raises((AssertionError, KeyError)):
        for seed in range(40):
            _pass(50, n, seed, **{left_out: False})
