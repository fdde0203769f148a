"""One section by pointers below slice 35: its children are read as they are
(one launch) or turned into ready records in a temporary first (two), by the
sizes of both.  Each choice, told apart by the launches, against the
one-thread-per-board kernel on child values drawn at random (both compute the
same function of any records).  Bit tables, compared exactly."""
import numpy as np
import pytest

from tests.gpu_helpers import ready, section_key, section_size

pytestmark = pytest.mark.gpu

RAW, READY = 1, 2  # launches


def _children(index, sec, n):
    """Per quadrant the number of the child section, or None."""
    out = []
    for q in range(4):
        bw = [list(x) for x in section_key(sec)]
        if sum(bw[q]) == 9:
            out.append(None)
            continue
        bw[q][n % 2] += 1  # black moves on an even number of stones
        out.append(index[tuple(map(tuple, bw))])
    return out


def _first(pp, n, holds):
    """The first section of slice n of which holds(boards, child values, walked
    states, lines) is true, and its children."""
    secs, _ = pp.slice_sections(n)
    above, _ = pp.slice_sections(n + 1)
    index = {section_key(s): i for i, s in enumerate(above)}
    for i, s in enumerate(secs):
        open_q = [q for q in range(4) if sum(section_key(s)[q]) < 9]
        if not open_q:
            continue
        walk = max(int(s["dim"][q]) for q in open_q)
        boards = section_size(s)
        kids = _children(index, s, n)
        values = sum(section_size(above[c]) for c in kids if c is not None)
        if holds(boards, values, walk, boards // walk):
            return secs, i, above, kids
    raise AssertionError(f"slice {n} has no such section")


def _check(n, holds, launches):
    import torch
    pp = ready()
    secs, i, above, kids = _first(pp, n, holds)
    boards = section_size(secs[i])
    gen = torch.Generator(device="cuda").manual_seed(n)
    offs, at = np.full(len(above), pp.PP_ABSENT, dtype=np.uint64), 0
    for c in kids:
        if c is not None:
            offs[c] = at
            at += section_size(above[c])
    values = torch.randint(-2**63, 2**63 - 1, (at, 8), dtype=torch.int64, device="cuda", generator=gen)
    children = [None if c is None else values[int(offs[c]):int(offs[c]) + section_size(above[c])] for c in kids]
    got = torch.zeros((boards + 1, 8), dtype=torch.int64, device="cuda")
    before = pp.launch_count()
    pp.section_compute(n, secs[i], children, got[:boards])
    assert pp.launch_count() - before == launches
    keep = np.zeros(len(secs), dtype=np.uint8)
    keep[i] = 1
    want = torch.zeros_like(got)
    plan = pp.SlicePlan(n, values, want[:boards], filter=keep, opts=(2, 0, 0, 2, 0), in_offsets=offs)
    plan.run()
    torch.cuda.synchronize()
    plan.close()
    assert torch.equal(got, want)  # the row past the section still zero


# the most child values a temporary is taken for, and one section above it
def test_temporary_is_bounded():
    _check(32, lambda boards, values, walk, lines: 2**25 < values <= 2 * boards < 2**27, RAW)


# children up to twice the boards, and more
@pytest.mark.parametrize("n, few, launches", [(33, True, READY), (30, True, READY), (30, False, RAW), (24, False, RAW)])
def test_children_against_boards(n, few, launches):
    _check(n, lambda boards, values, walk, lines:
           20_000 < boards < 2_000_000 and walk >= 64 and (values <= 2 * boards) == few, launches)


# short lines, few lines of medium length; many of them, and longer ones
@pytest.mark.parametrize("n, holds, launches", [
    (34, lambda boards, values, walk, lines: walk == 3 and lines == 3, RAW),
    (34, lambda boards, values, walk, lines: walk == 3 and lines > 1000, RAW),
    (34, lambda boards, values, walk, lines: walk == 10 and 100 < lines <= 256, RAW),
    (34, lambda boards, values, walk, lines: walk == 10 and lines > 256, READY),
    (34, lambda boards, values, walk, lines: walk == 18 and lines < 32, READY),
    (33, lambda boards, values, walk, lines: walk == 10 and lines < 32, RAW),
])
def test_short_walks_read_the_children_as_they_are(n, holds, launches):
    _check(n, lambda boards, values, walk, lines: values <= 2 * boards and holds(boards, values, walk, lines), launches)
