"""CPU models of how the recursion kernels walk (csrc/delta_column.cu): the warps' first tasks, the column kernels' four
rows a step with their chunks of coefficients and flushes of the transposition block, and the four-row degree-lane kernel
with its loads issued four rows ahead.  (The values, row after row, are modelled in test_column_schedule.py.)"""
import pytest

WARPS = 8


@pytest.mark.parametrize("sms,per", [(152, 1), (152, 2), (152, 3), (152, 4), (148, 3), (1, 2)])
def test_first_tasks_are_all_different_and_spread(sms, per):
    """next_task: task n goes to CTA n mod grid, and CTAs that share an SM start with different warps."""
    grid = sms * per
    first = {(b, w): ((w - b // sms) & (WARPS - 1)) * grid + b for b in range(grid) for w in range(WARPS)}
    assert sorted(first.values()) == list(range(grid * WARPS))  # later ones follow from the counter
    for sm in range(sms):
        starts = [next(w for w in range(WARPS) if first[(b, w)] < grid) for b in range(sm, grid, sms)]
        assert len(set(starts)) == len(starts)


def column_walk(l, m0, four):
    """Rows in the order the kernels write them, the chunk that serves each, and the flushed chunks with the rows staged
    before them; four: the four-row step (four rows 4k + 3 .. 4k)."""
    rows, flushes, staged, chunk, mp = [], [], set(), None, l
    while mp >= m0:
        j = mp & 31
        if mp == l or j == 31:
            chunk = mp & ~31
        n = 4 if four and (mp & 3) == 3 else 1
        for k in range(n):
            assert j - k >= 0 and (mp - k) & ~31 == chunk
            rows.append(mp - k)
            if mp - k >= m0 + 32:
                staged.add(mp - k)
        low = mp - n + 1
        if low & 31 == 0 and low >= m0 + 32:
            flushes.append((low, frozenset(staged)))
            staged = set()
        mp -= n
    return rows, flushes, staged


@pytest.mark.parametrize("four", [False, True])
@pytest.mark.parametrize("l", [0, 1, 2, 3, 4, 31, 32, 33, 35, 63, 64, 66, 95, 100, 127, 128, 200, 255])
def test_column_walk_takes_every_row_and_flushes_whole_chunks(l, four):
    for m0 in range(0, l + 1, 32):
        rows, flushes, left = column_walk(l, m0, four)
        # the last four rows end at m0, a multiple of 32, so that none lies below it
        assert rows == list(range(l, m0 - 1, -1))
        assert not left
        assert [c for c, _ in flushes] == [c for c in range(l & ~31, m0 + 31, -32)]
        for c, staged in flushes:
            assert staged == set(range(c, min(l, c + 31) + 1))


def tri_idx(r, l, L):
    return r * L - r * (r - 1) // 2 + (l - r)


@pytest.mark.parametrize("L", [1, 2, 5, 31, 32, 33, 64, 130, 161, 257])
def test_four_row_degree_lane_walk(L):
    """lane_recursion_deep_kernel: each row m' = top .. m of a task once, with the loads of its own row in its slot, the tile
    of its own row block, and the four-row step only where every degree of the warp is under way."""
    nI, D = (L + 127) // 128, 4
    ibase = {(r, i): 1000 * r + i for r in range(L) for i in range(nI)}
    for m in sorted({0, 1, 2, 31, 32, L // 2, L - 2, L - 1} & set(range(L))):
        for kc in range(m // 32, (L + 31) // 32):
            top = min(32 * kc + 31, L - 1)
            lane = min(31, L - 1 - 32 * kc)  # one lane's addresses stand for all: they differ by l
            l = 32 * kc + lane
            ask, kidx, ibr = top, top * L - top * (top - 1) // 2 + (l - top), (top, m >> 7)
            slots = [None] * D

            def fetch(q):
                nonlocal ask, kidx, ibr
                slots[q] = None
                if ask >= m:
                    slots[q] = (ask, kidx if ask <= l else None, ibase[ibr])
                    ask -= 1
                    kidx -= L - (ask + 1)
                    ibr = (ibr[0] - 1, ibr[1])

            for q in range(D):
                fetch(q)
            tb, tbn, mp, done = None, ibase[(m, top >> 7)], top, []

            def row(q):
                assert slots[q][0] == mp - (q if four else 0)
                r = slots[q][0]
                if r <= l:
                    assert slots[q][1] == tri_idx(r, l, L) and 0 <= slots[q][1] < L * (L + 1) // 2
                assert slots[q][2] == ibase[(r, m >> 7)]
                assert tb == ibase[(m, r >> 7)] + kc
                done.append(r)

            while mp >= m:
                four = mp < 32 * kc and mp - 3 > m and (mp & 127) != 127 and (mp >> 7) == ((mp - 3) >> 7)
                if four:
                    for q in range(D):
                        row(q)
                    for q in range(D):
                        fetch(q)
                    mp -= D
                    continue
                for q in range(D):
                    if mp >= m:
                        if mp == top or (mp & 127) == 127:
                            tb = tbn + kc
                            if mp >> 7:
                                tbn = ibase[(m, (mp >> 7) - 1)]
                        row(q)
                        fetch(q)
                        mp -= 1
            assert done == list(range(top, m - 1, -1))
