"""Which neighbours a run of the row-run sweep form waits for, against brute force.

The row-run form scores consecutive classes (u, v0..v0+n-1) of one class row
at once.  An update may only be decided when every earlier update of the
raster scan whose window overlaps its own is done.  The kernel waits, per
neighbour tile, for: the right tile's classes of this row before the run's
last one; the left and the three lower tiles' previous class rows; the three
upper tiles' previous sweep.  Here every pair of overlapping windows of two
sweeps is listed and checked against those rules, and -- the rules being no
wider than needed -- each rule is met with equality by some pair.
"""
import itertools

import pytest


def _kind(di, dj):
    return "sweep" if di < 0 else "right" if (di == 0 and dj > 0) else "row"


@pytest.mark.parametrize("S,L", [(3, 3), (4, 3), (5, 5), (7, 5)])
def test_waits_cover_every_earlier_overlapping_update(S, L):
    tight = set()
    steps = list(itertools.product(range(2), range(S), range(S)))   # (sweep, u, v) in raster order
    for di, dj in itertools.product((-2, -1, 0, 1, 2), repeat=2):
        if (di, dj) == (0, 0):
            continue
        for (s, u, v), (s2, u2, v2) in itertools.product(steps, steps):
            if (s2, u2, v2) >= (s, u, v):
                continue
            if abs(di * S + u2 - u) >= L or abs(dj * S + v2 - v) >= L:
                continue   # the two windows share no camera pixel
            assert max(abs(di), abs(dj)) == 1, "only adjacent patches' windows overlap"
            kind = _kind(di, dj)
            done = s2 * S * S + u2 * S + v2 + 1                      # steps the neighbour must have finished
            if kind == "right":
                need = s * S * S + u * S + v                         # its classes of this row before v
            elif kind == "row":
                need = s * S * S + u * S
            else:
                need = s * S * S
            assert done <= need, (kind, di, dj, (s, u, v), (s2, u2, v2))
            if done == need:
                tight.add(kind)
    if S == L:
        assert tight == {"right", "row", "sweep"}


@pytest.mark.parametrize("S,L", [(3, 3), (5, 5), (7, 5)])
def test_a_run_may_overlap_only_its_right_neighbours_same_run(S, L):
    # within one class row, the only windows of another patch that overlap an
    # update's are the right patch's at smaller v: a tile's patches are taken
    # from right to left, and a run is final once the right tile's run is
    for u, v, v2 in itertools.product(range(S), repeat=3):
        for di, dj in itertools.product((-1, 0, 1), repeat=2):
            if (di, dj) == (0, 0):
                continue
            overlap = abs(di * S) < L and abs(dj * S + v2 - v) < L
            assert not overlap or (di == 0 and (dj == 1 and v2 < v or dj == -1 and v2 > v))
