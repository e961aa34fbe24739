"""Model check of the ring protocol of the FP32 march kernel (NS recursion steps
per launch).

Set i (V_m row i + 2, set 0 rows 0, 1, 2; V_{m-1} row i; entries row i) lands on
full[i]; done_s[i] completes when every warp of stage s and the warp of the
moment sums have finished row i.  Stage s at row i reads its input rows
i .. i + 2 (its own registers keep rows i and i + 1), entries row i + s, and as
subtrahend row i (stage 0) or row i + 2 of the ring that stage s - 1 reads; it
writes row i of its output ring.  The moment sums of stage s read input rows
i .. i + 2 in shared memory.  The producer issues set i after the last stage
has finished row i - lag (before that row exists: an earlier stage the rows it
leads by).  Barriers are rings of BARS phases whose waits test a parity only.

The test replays these rules with the kernel's ring sizes under random
interleavings and checks that every read finds the row it wants, that no ring
row in flight or still to be read is overwritten, that no barrier runs two
phases ahead of a waiter, and that all rows are done.
"""
import random

import pytest

BARS = 16
ROWS = 8


def _sizes(ns, lag):
    if ns == 1:
        return dict(v=lag + 2, p=lag, s=ROWS, c=lag)
    return dict(v=ROWS, p=ROWS, s=ROWS, c=ROWS)


class _Bar:
    def __init__(self):
        self.done = -1      # last completed row of the slot's barrier, by row

    def completed(self, row):
        assert self.done - row < 2 * BARS - (BARS - 1), "a barrier ran two phases ahead of its waiter"
        return self.done >= row


def _run(ns, lag, nrow, seed, size=None):
    rng = random.Random(seed)
    last = ns - 1
    n = size or _sizes(ns, lag)
    rows = [nrow + 2 * (last - s) for s in range(ns)]
    full = [_Bar() for _ in range(BARS)]
    done = [[_Bar() for _ in range(BARS)] for _ in range(ns)]
    ring = dict(v=[None] * n["v"], p=[None] * n["p"], c=[None] * n["c"])
    for s in range(last):
        ring["s%d" % s] = [None] * n["s"]
    busy = {}               # (ring, slot) -> readers that have not finished

    def full_ok(i):
        return full[i % BARS].completed(i)

    def done_ok(s, i):
        return done[s][i % BARS].completed(i)

    def put(name, row):
        slot = row % len(ring[name])
        assert not busy.get((name, slot)), f"{name} row {ring[name][slot]} overwritten by {row} while it is read"
        assert ring[name][slot] != ("in flight",), "a copy in flight overwritten"
        ring[name][slot] = row

    def get(name, row):
        slot = row % len(ring[name])
        assert ring[name][slot] == row, f"{name}: wanted row {row}, found {ring[name][slot]}"
        return (name, slot)

    def inputs(s):
        return "v" if s == 0 else "s%d" % (s - 1)

    def rows_read(actor, i):
        if actor[0] == "sums":
            s = actor[1]
            return [(inputs(s), i + d) for d in range(3)]
        s = actor[1]
        got = [(inputs(s), r) for r in ([0, 1, 2] if i == 0 else [i + 2])] + [("c", i + s)]
        got.append(("p", i) if s == 0 else (inputs(s - 1), i + 2))
        return got

    # two warps per stage stand for its warps; one warp for the sums of all stages
    actors = [("stage", s, k) for s in range(ns) for k in range(2)]
    state = {a: [0, "wait"] for a in actors}
    order = [(s, t - 2 * s) for t in range(rows[0]) for s in range(ns) if 0 <= t - 2 * s < rows[s]]
    sums = [0, "wait"]
    issued, flight = 0, []
    arrived = {}

    def arrive(s, i):
        arrived[s, i] = arrived.get((s, i), 0) + 1
        if arrived[s, i] == 3:
            b = done[s][i % BARS]
            assert b.done == i - BARS or (b.done == -1 and i < BARS), "phases out of order"
            b.done = i

    for _ in range(10 ** 6):
        moves = [a for a in actors if state[a][0] < rows[a[1]]]
        if sums[0] < len(order):
            moves.append("sums")
        if issued < rows[0]:
            moves.append("producer")
        if flight:
            moves.append("land")
        if not moves:
            return
        m = rng.choice(moves)
        if m == "producer":
            s, r = last, issued - lag
            while r < 0 and s > 0:
                r, s = r + 2, s - 1
            if r >= 0 and not done_ok(s, r):
                continue
            for name, row in [("v", q) for q in ([0, 1, 2] if issued == 0 else [issued + 2])] + [("p", issued),
                                                                                                 ("c", issued)]:
                put(name, row)
                ring[name][row % len(ring[name])] = ("in flight",)
            flight.append(issued)
            issued += 1
        elif m == "land":
            i = flight.pop(rng.randrange(len(flight)))
            for name, row in [("v", q) for q in ([0, 1, 2] if i == 0 else [i + 2])] + [("p", i), ("c", i)]:
                ring[name][row % len(ring[name])] = row
            b = full[i % BARS]
            assert b.done == i - BARS or (b.done == -1 and i < BARS), "a set landed out of phase"
            b.done = i
        elif m == "sums":
            s, i = order[sums[0]]
            if sums[1] == "wait":
                if full_ok(i) if s == 0 else done_ok(s - 1, i + 2):
                    for name, row in rows_read(("sums", s), i):
                        busy.setdefault(get(name, row), set()).add(("sums", s, i))
                    sums[1] = "read"
            else:
                for name, row in rows_read(("sums", s), i):
                    busy[get(name, row)].discard(("sums", s, i))
                arrive(s, i)
                sums[:] = [sums[0] + 1, "wait"]
        else:
            s, (i, st) = m[1], state[m]
            if st == "wait":
                ok = full_ok(i) if s == 0 else done_ok(s - 1, i + 2)
                if ok and s < last and i >= n["s"]:
                    f = i - n["s"]
                    two = s + 2 <= last and f >= 2
                    ok = done_ok(s + 2, f - 2) if two else done_ok(s + 1, f)
                if ok:
                    for name, row in rows_read(m, i):
                        busy.setdefault(get(name, row), set()).add((m, i))
                    state[m][1] = "write"
            else:
                for name, row in rows_read(m, i):
                    busy[get(name, row)].discard((m, i))
                if s < last:
                    slot = i % n["s"]
                    assert not busy.get(("s%d" % s, slot)), "a stage's row overwritten while it is read"
                    ring["s%d" % s][slot] = i
                arrive(s, i)
                state[m] = [i + 1, "wait"]
    raise AssertionError("no progress: the protocol deadlocks")


@pytest.mark.parametrize("ns,lag", [(1, 3), (1, 5), (1, 6), (1, 8), (2, 8), (3, 8)])
@pytest.mark.parametrize("nrow", [1, 2, 3, 7, 12, 40])
def test_march_protocol_random_schedules(ns, lag, nrow):
    for seed in range(8):
        _run(ns, lag, nrow, seed)


@pytest.mark.parametrize("ns,lag,ring,rows", [(1, 6, "v", 7), (2, 8, "v", 7), (2, 8, "p", 5), (2, 8, "c", 6)])
def test_a_ring_row_too_few_is_caught(ns, lag, ring, rows):
    size = dict(_sizes(ns, lag), **{ring: rows})
    with pytest.raises(AssertionError):
        for seed in range(40):
            _run(ns, lag, 40, seed, size)
