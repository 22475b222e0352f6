"""What the kernel skips of the tile program (levels 18 and 20): in FP64 the
words past a slab's longest record, and the weights of its leading chunks."""
import os
import sys

import pytest

PKG = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_00193_gb300")
sys.path.insert(0, PKG)
import basisgen  # noqa: E402


@pytest.mark.parametrize("level", [18, 20])
def test_work_covers_the_program(level):
    tp = basisgen.TileProgram(basisgen.Level(level))
    words, slabs, off = tp.encode()
    pad = tp.zero | tp.zero << 13
    assert len(tp.work) == len(slabs) == off[-1]
    seen = 0
    for (first, meta), (terms, unit) in zip(slabs, tp.work):
        assert (terms + 4) >> 2 == meta >> 1 and 0 <= unit <= meta >> 1 and (unit == meta >> 1) == bool(meta & 1)
        for lane in range(basisgen.TILE_LANES):
            for q in range(meta >> 1):
                at = 4 * (first + q * basisgen.TILE_LANES + lane)
                for i in range(4):
                    k = 4 * q + i - 1                       # index of the term, -1: the head
                    if k < 0:
                        continue
                    t = words[at + i]
                    assert k < terms or t == pad            # nothing past the longest record
                    assert q >= unit or tp.weights[t >> 26] == 1
                    seen += t != pad
    assert seen == sum(len(t) for ph in tp.phases for _, _, t in ph)


def visited(bounds, first, last, warps, warp):
    """The slabs that a warp runs, stepped as the kernel does: the successor is chosen one slab ahead, across
    the end of the phase."""
    out, total = [], len(bounds) - 1
    start, end, s, ns, ready = bounds[first], bounds[first + 1], 0, 0, False
    for p in range(first, last):
        after = bounds[min(p + 2, total)]
        if not ready:
            s = start + warp
            ns = s + warps if s + warps < end else end + warp
        ready = s < end
        while s < end:
            stop = end if ns < end else after
            out.append((p, s))
            s, ns = ns, ns + warps if ns + warps < stop else stop + warp
        start, end = end, after
    return out


@pytest.mark.parametrize("warps", [1, 4, 32])
def test_each_slab_runs_once_in_its_phase(warps):
    import random
    rnd = random.Random(warps)
    programs = [basisgen.TileProgram(basisgen.Level(18)).encode()[2]]
    for _ in range(300):
        b = [0]
        for _ in range(rnd.randint(1, 8)):
            b.append(b[-1] + rnd.choice([0, 1, warps - 1, warps, warps + 1, 3 * warps + 2]))
        programs.append(b)
    for b in programs:
        cut = rnd.randint(0, len(b) - 1)
        for lo, hi in ((0, cut), (cut, len(b) - 1)):
            if lo < hi:
                got = sorted(sum((visited(b, lo, hi, warps, w) for w in range(warps)), []))
                assert got == [(p, s) for p in range(lo, hi) for s in range(b[p], b[p + 1])]
