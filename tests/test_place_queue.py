"""The queue of straddling rows in rank_count_kernel (csrc/fusion.cu): whether
a block empties it after a tile has to be the same in all of its warps, since
the emptying holds barriers.  Every interleaving of two warps over a few tiles
on the CPU, with the decision taken from the count read after the tile's
barrier (warps can differ) and from a count read before it and combined by it
(they cannot, and the block knows exactly)."""
import os

import pytest

LIMIT = 3


def _disagreements(adds, before_barrier):
    """adds[t][w]: what warp w adds in tile t -> the number of reachable ends
    of a tile where the warps decide differently, or not by the tile's count."""
    tiles, warps = len(adds), len(adds[0])
    bad, seen = 0, set()
    # per warp: (tile, step); step 0: add, 1: read (before), 2: at the barrier, 3: read (after)
    start = (tuple((0, 0) for _ in range(warps)), 0, tuple(() for _ in range(warps)),
             tuple(0 for _ in range(warps)))
    todo = [start]
    while todo:
        state = todo.pop()
        if state in seen:
            continue
        seen.add(state)
        pos, count, decided, read = state
        moved = []
        for w in range(warps):
            t, step = pos[w]
            if t == tiles:
                continue
            p, c, d, r = list(pos), count, list(decided), list(read)
            if step == 0:
                c += adds[t][w]
                p[w] = (t, 1)
            elif step == 1:
                r[w] = c
                p[w] = (t, 2)
            elif step == 2:
                continue
            else:
                d[w] = d[w] + (c > LIMIT,)
                p[w] = (t + 1, 0)
            moved.append((tuple(p), c, tuple(d), tuple(r)))
        if all(step == 2 and t < tiles for t, step in pos) and len({t for t, _ in pos}) == 1:
            t = pos[0][0]
            if before_barrier:   # the barrier combines the counts read before it
                full = any(v > LIMIT for v in read)
                bad += full != (count > LIMIT)
                moved.append((tuple((t + 1, 0) for _ in pos), count,
                              tuple(d + (full,) for d in decided), read))
            else:
                moved.append((tuple((t, 3) for _ in pos), count, decided, read))
        done = min(len(d) for d in decided)
        if any(len({d[t] for d in decided}) > 1 for t in range(done)):
            bad += 1
            continue
        todo += moved
    return bad


# counts that stay below the limit, reach it, and pass it in each of the tiles
# (the emptying itself is left out: it begins and ends with barriers)
@pytest.mark.parametrize("adds", [
    ((1, 1), (1, 1), (0, 0)), ((2, 1), (1, 0), (1, 0)), ((0, 3), (0, 1), (1, 1)), ((4, 0), (1, 1))])
def test_the_block_decides_as_one(adds):
    assert _disagreements(adds, before_barrier=True) == 0


def test_a_count_read_after_the_barrier_can_split_the_block():
    assert _disagreements(((2, 1), (1, 0)), before_barrier=False) > 0


def test_the_kernel_decides_at_the_barrier():
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    text = open(os.path.join(root, "paper_2608_07152_gb300", "csrc", "fusion.cu")).read()
    body = text[text.index("rank_count_kernel("):]
    body = body[:body.index("\n}\n")]
    assert "__syncthreads_or(*reinterpret_cast<volatile int*>(&q_n)" in body
    # no decision from a count read after a barrier
    assert "if (n > kPlaceQueue" not in body and "(q_n > kPlaceQueue" not in body
