"""The staging-tile protocol of the streaming attention kernel, explored exhaustively on the CPU.

Four warps share a lane quarter's two staging tiles.  Only warp 0 waits for the others ("the tile is written") before it
stores a tile, so the warps may run apart; this walks through every interleaving of their steps with the barrier mapping
that the kernel's source states and checks that no tile is stored before all four warps have written it.
"""
import os
import re

import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_14107_b200", "csrc", "attn_stream.cuh")
WARPS = 4


def mapping():
    text = open(SRC).read()

    def fn(name):
        expr = re.search(r"constexpr \w+ %s\(int j\) \{ return ([^;]+); \}" % name, text).group(1)
        return eval("lambda j: " + expr)
    return fn("written_bar"), fn("written_parity")


def explore(bar, parity, tiles):
    """First tile that some interleaving stores before it is written (None: there is none); also checks that the kernel
    cannot get stuck.  A warp's steps per tile: 0 hand P over (its buffer is free once all four have handed over the previous
    one's), [1 request the rows of the next tile (warp 0), ] wait for the rows of this tile, 2 write it and arrive, [3 wait
    for the arrivals and store (warp 0)]."""
    last = {0: 3, 1: 2, 2: 2, 3: 2}
    start = ((0, 0),) * WARPS                      # per warp: (tile, next step)
    seen, todo, finished = {start}, [start], False
    passed = lambda st, w, j, step: st[w] > (j, step)      # warp w has taken that step of tile j
    while todo:
        st = todo.pop()
        if all(j == tiles for j, _ in st):
            finished = True
            continue
        moved = False
        for w, (j, step) in enumerate(st):
            if j == tiles:
                continue
            if step == 0 and j > 0 and not all(passed(st, v, j - 1, 0) for v in range(WARPS)):
                continue
            if step == 2 and not (j < 2 or passed(st, 0, j - 1, 1)):       # rows of tiles 0 and 1 are requested up front
                continue
            if step == 3:
                arrivals = sum(1 for v in range(WARPS) for t in range(tiles) if bar(t) == bar(j) and passed(st, v, t, 2))
                if (arrivals // WARPS) & 1 == parity(j):                   # the phase waited for has not completed
                    continue
                if not all(passed(st, v, j, 2) for v in range(WARPS)):
                    return j, finished
            nxt = step + 1 if not (w > 0 and step == 0) else 2
            new = (j, nxt) if nxt <= last[w] else (j + 1, 0)
            s2 = st[:w] + (new,) + st[w + 1:]
            moved = True
            if s2 not in seen:
                seen.add(s2)
                todo.append(s2)
        assert moved, f"stuck at {st}"
    return None, finished


@pytest.mark.parametrize("tiles", [1, 2, 3, 6])
def test_no_tile_is_stored_before_its_four_warps_have_written_it(tiles):
    bar, parity = mapping()
    assert explore(bar, parity, tiles) == (None, True)


def test_one_barrier_for_both_staging_tiles_is_not_enough():
    # the exploration itself: with a single barrier a fast warp's arrival for the next tile stands in for a slow warp's
    early, _ = explore(lambda j: 0, lambda j: j & 1, 3)
    assert early is not None
