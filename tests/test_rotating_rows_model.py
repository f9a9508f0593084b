"""Why a warp of the 4096 < d' <= 8192 kernel (gbs_tc_uv2.cu) whose bounded wait ran out walks on instead of leaving: a host model of
one token's warps, their lane quadrants' rows moving on from tile to tile, the barrier that joins the warps with rows in a tile,
and the block's closing barrier.  No GPU wait is made to run out: the model is what can be tested of it."""
import pytest

STAGES = 4


def ends(slabs, n_tiles, failing, walk_on):
    """Whether every warp reaches the closing barrier.  A warp is (quadrant, half); `failing` is (warp, tile of its expired wait)."""
    warps = [(q, h) for q in range(4) for h in range(2)]

    def plan_of(w):                                   # the tiles in which this warp has rows
        return [it for it in range(n_tiles) if slabs == 4 or (w[0] - it) % 4 < slabs]

    todo = {w: plan_of(w) for w in warps}
    dead = {w: False for w in warps}
    gone, at = set(), {}                              # warps at the closing barrier; barrier (tile) a warp waits at
    arrived, poisoned = {}, set()
    for _ in range(100 * n_tiles):
        moved = False
        for w in warps:
            if w in gone:
                continue
            if w in at:                               # waits until all the tile's warps have come
                it = at[w]
                if len(arrived[it]) < 2 * slabs:
                    continue
                del at[w]
                moved = True
                if it in poisoned:
                    dead[w] = True
                    if not walk_on:
                        gone.add(w)
                continue
            moved = True
            if not todo[w]:
                gone.add(w)
                continue
            it = todo[w].pop(0)
            if (w, it) == failing:
                dead[w] = True
            if dead[w]:
                poisoned.add(it)
            arrived.setdefault(it, set()).add(w)
            at[w] = it
        if not moved:
            break
    return len(gone) == len(warps)


@pytest.mark.parametrize("slabs", [3, 4])
def test_every_warp_reaches_the_end_if_it_walks_on(slabs):
    for n_tiles in (1, 2, 5, 9):
        assert ends(slabs, n_tiles, None, True)
        for q in range(4):
            for h in range(2):
                for it in range(n_tiles):
                    assert ends(slabs, n_tiles, ((q, h), it), True)


def test_leaving_leaves_the_resting_warps_behind():
    assert ends(4, 9, ((1, 0), 3), False)             # no warp rests: all see it
    assert not ends(3, 9, ((1, 0), 3), False)
