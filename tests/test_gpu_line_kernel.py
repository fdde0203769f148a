"""The line kernel over ready children against the one-thread-per-board
kernel, on child values drawn at random (both compute the same function of
any records): every line axis and every arrangement of empty quadrants,
sections of a few lines, partly filled lane groups, and ranges of states
split over several blocks.  The values are bit tables, compared exactly."""
import numpy as np
import pytest

from tests.gpu_helpers import ready, section_key, section_size

pytestmark = pytest.mark.gpu


def _shape(s):
    """(line axis, the other quadrants with empty cells): the longest lines,
    the higher quadrant of equals."""
    open_q = [q for q in range(4) if sum(section_key(s)[q]) < 9]
    axis = max(open_q, key=lambda q: (int(s["dim"][q]), q))
    return axis, tuple(q for q in open_q if q != axis)


def _sample(pp, n, limit):
    """Per shape the smallest section, the first whose lines do not fill the
    last lane group, and the largest of at most `limit` boards."""
    secs, _ = pp.slice_sections(n)
    by = {}
    for i, s in enumerate(secs):
        if section_size(s) <= limit:
            by.setdefault(_shape(s), []).append(i)
    keep = np.zeros(len(secs), dtype=np.uint8)
    for (axis, _), group in by.items():
        group.sort(key=lambda i: section_size(secs[i]))
        keep[group[0]] = keep[group[-1]] = 1
        ragged = [i for i in group if section_size(secs[i]) // int(secs[i]["dim"][axis]) % 32]
        if ragged:
            keep[ragged[len(ragged) // 2]] = 1
    return secs, keep


# slice 34 has every (axis, one other) shape, 33 and 30 several others, 24
# quadrants with many empty cells (long move lists)
@pytest.mark.parametrize("n, limit", [(34, 60_000), (33, 40_000), (30, 60_000), (24, 300_000)])
def test_lines_equal_per_board(n, limit):
    import torch
    pp = ready()
    secs, keep = _sample(pp, n, limit)
    assert keep.any()
    above, _ = pp.slice_sections(n + 1)
    offs, at = np.full(len(above), pp.PP_ABSENT, dtype=np.uint64), 0
    for i in np.flatnonzero(pp.slice_children(n, keep)):
        offs[i] = at
        at += section_size(above[i])
    gen = torch.Generator(device="cuda").manual_seed(n)
    kids = torch.randint(-2**63, 2**63 - 1, (at, 8), dtype=torch.int64, device="cuda", generator=gen)
    total = int(sum(section_size(s) for s, k in zip(secs, keep) if k))
    outs = []
    for stage in (1, 2):
        out = torch.zeros((total + 1, 8), dtype=torch.int64, device="cuda")
        plan = pp.SlicePlan(n, kids, out, filter=keep, opts=(2, 0, 0, stage, 0), in_offsets=offs)
        plan.set_prepared(2)
        plan.run()
        torch.cuda.synchronize()
        plan.close()
        assert not bool(out[total].any())  # nothing past the kept sections
        outs.append(out)
    assert torch.equal(outs[0], outs[1])
