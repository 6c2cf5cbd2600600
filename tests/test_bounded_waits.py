"""The gathering warps of the one-stage contraction kernel wait for a tile's buffer with a limit and meet at a barrier that has
none.  A model of both: the buffer's barrier completes at some moment, every warp polls at moments of its own, gives up behind
its limit or once another warp has, and then either leaves or comes to the barrier.  However the outcomes differ between the
warps, all of them must get out."""
import itertools

WARPS, LIMIT, TILES = 3, 2, 3


def _stuck(leave_alone, outcomes):
    """outcomes[tile][warp]: did that warp's wait succeed?  Returns whether a warp is left in the barrier for ever."""
    inside = set(range(WARPS))
    for tile in outcomes:
        if not inside:
            return False
        arrived = {w for w in inside if tile[w] or not leave_alone}
        # the barrier counts all warps: it opens only if every one of them arrives
        if arrived and len(arrived) < WARPS:
            return True
        if leave_alone:
            inside = arrived
        elif not all(tile[w] for w in inside):
            inside = set()                                     # the barrier's answer is the same for all: they leave together
    return False


def _all_outcomes():
    """Every outcome that polls at arbitrary moments can give: the barrier completes at moment c, warp w polls LIMIT times from
    its own moment on, testing the barrier before the flag that another warp sets when it gives up."""
    per_tile = set()
    for c in range(6):
        for starts in itertools.product(range(4), repeat=WARPS):
            polls = sorted((s + i, w) for w, s in enumerate(starts) for i in range(LIMIT))
            ok, failed, tries = {}, False, [0] * WARPS
            for moment, w in polls:
                if w in ok:
                    continue
                tries[w] += 1
                if moment >= c:
                    ok[w] = True
                elif failed or tries[w] == LIMIT:
                    ok[w], failed = False, True
            per_tile.add(tuple(ok[w] for w in range(WARPS)))
    return itertools.product(sorted(per_tile), repeat=TILES)


def test_warps_that_decide_alone_can_be_left_behind():
    assert any(_stuck(True, o) for o in _all_outcomes())


def test_warps_that_agree_at_the_barrier_all_leave():
    assert not any(_stuck(False, o) for o in _all_outcomes())


def test_the_kernel_agrees_at_the_barrier():
    """The code of the loop: no way out between the wait and the barrier, and out of the barrier only by its common answer."""
    import os
    import re
    src = open(os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1711_01348_b200", "csrc", "mma.cu")).read()
    loop = src[src.index("// ---- gathering warps ----"):src.index("// ---- epilogue warps")]
    loop = loop[loop.index("for (int t = 0; t < n_tiles"):]
    between = loop[loop.index("mbar_wait("):loop.index("any_of_warps<CT>(!ok)")]
    assert not re.search(r"\b(break|return|goto)\b", re.sub(r"//.*", "", between))
    assert "bar.sync" not in loop
