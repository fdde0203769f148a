"""How a midgame plan arranges its boards: in packs, one by one, or both,
beside each other or one after the other.  What was chosen is told apart by
the launches of a run; the values are the oracle's (stored ones for 12 empty
cells), or those of single boards a level at a time.  Bit tables, compared
exactly."""
import numpy as np
import pytest

from paper_1404_0743_gb300 import inputs
from tests.gpu_helpers import midgame_oracle, ready, to_host
from tests.test_gpu_midgame import _golden
from tests.test_gpu_parity import class_mask

pytestmark = pytest.mark.gpu


def _stored(count):
    """The first boards of the 1024 x 12 workload and their stored values."""
    rows = list(_golden())[:count]
    assert [i for i, _, _ in rows] == list(range(count))
    return inputs.batched_midgame_boards(1024)[:count], np.array([w for _, _, w in rows], dtype=np.uint64)


def _drawn(specs, seed):
    return np.concatenate([inputs.midgame_boards(n, k, seed + 1000 * k) for n, k in specs])


def _run(boards, kmax, mode, parity, launches=None):
    import torch
    pp = ready()
    plan = pp.MidgamePlan(boards, kmax)
    plan.set_parity(parity)
    plan.configure(mode)
    ws = torch.empty(pp.midgame_workspace_bytes(len(boards), kmax), dtype=torch.uint8, device="cuda")
    out = torch.full((len(boards), 8), -1, dtype=torch.int64, device="cuda")
    plan.run(ws, out)
    before = pp.launch_count()
    plan.run(ws, out)  # the second run finds the tables of the first
    took = pp.launch_count() - before
    plan.status()
    got = to_host(out)
    plan.close()
    assert launches is None or took == launches
    return got


def _of_class(values, parity):
    return values if parity < 0 else values & class_mask(parity)


# launches: masks and levels of either kind (persistent: one launch of levels;
# both kinds in one where few fills are left over), the packs' roots where a
# level is a launch, one for the boards of at most 7 empty cells
@pytest.fixture(scope="module")
def shapes():
    """Packs of two shapes, other shapes left over, boards solved in one block,
    shuffled."""
    twelve, values = _stored(48)
    others = _drawn(((32, 10), (5, 9), (3, 8), (17, 6)), 0xA44A)
    order = np.random.default_rng(9).permutation(48 + len(others))
    return np.concatenate([twelve, others])[order], np.concatenate([values, midgame_oracle(others)])[order]


@pytest.mark.parametrize("mode, launches", [(1, 2 + 1 + 1), (2, (1 + 13 + 1) + (1 + 10) + 1), (3, (1 + 13 + 1) + (1 + 10) + 1)])
@pytest.mark.parametrize("parity", [-1, 0, 1])
def test_packs_of_two_shapes_beside_single_boards(shapes, mode, launches, parity):
    boards, want = shapes
    assert (_run(boards, 12, mode, parity, launches) == _of_class(want, parity)).all()


@pytest.mark.parametrize("mode, launches", [(1, 2), (2, 1 + 10 + 1), (3, 1 + 10 + 1)])
@pytest.mark.parametrize("parity", [-1, 0, 1])
def test_packs_of_two_shapes_alone(mode, launches, parity):
    boards = _drawn(((16, 8), (16, 9)), 0xA44B)
    assert (_run(boards, 9, mode, parity, launches) == _of_class(midgame_oracle(boards), parity)).all()


@pytest.mark.parametrize("mode, launches", [(1, 2), (2, 1 + 11), (3, 1 + 11)])
def test_single_boards_of_unequal_shapes(mode, launches):
    boards = _drawn([(6, k) for k in (8, 9, 10)], 0xA44C)
    assert (_run(boards, 10, mode, -1, launches) == midgame_oracle(boards)).all()


# packed twelve-cell boards beside four with 14: 16 of them don't win their
# second kind of levels back (whole tables), 64 do, but not with the four at
# their occupancy
@pytest.mark.parametrize("packed, mode, parity, launches", [
    (16, 1, -1, 2), (16, 1, 0, 3), (16, 2, -1, 1 + 15), (16, 3, 1, 1 + 15), (64, 1, -1, 4), (64, 1, 1, 3),
    (64, 2, -1, (1 + 13 + 1) + (1 + 15))])
def test_choice_by_the_fills_left_over(packed, mode, parity, launches):
    twelve, values = _stored(packed)
    deep = _drawn(((4, 14),), 0xA44D)
    want = np.concatenate([values, np.concatenate([_run(deep[i:i + 1], 14, 2, -1) for i in range(4)])])
    boards = np.concatenate([deep, twelve])
    want = np.concatenate([want[packed:], want[:packed]])
    assert (_run(boards, 14, mode, parity, launches) == _of_class(want, parity)).all()


# one shape, its last 15 boards left over
@pytest.mark.parametrize("parity, launches", [(-1, 2), (0, 3)])
def test_one_shape_with_as_many_left_over(parity, launches):
    boards = inputs.midgame_boards(31, 13, 0xA451)
    want = np.concatenate([_run(boards[i:i + 8], 13, 2, parity) for i in range(0, 31, 8)])
    assert (_run(boards, 13, 1, parity, launches) == want).all()


def test_one_plan_through_every_mode_and_class():
    """A plan that holds both arrangements takes each by the mode and class
    set last."""
    import torch
    pp = ready()
    twelve, values = _stored(20)  # 16 in a pack, 4 left over
    plan = pp.MidgamePlan(twelve, 12)
    ws = torch.empty(pp.midgame_workspace_bytes(20, 12), dtype=torch.uint8, device="cuda")
    out = torch.zeros((20, 8), dtype=torch.int64, device="cuda")
    for mode, parity in ((1, -1), (3, -1), (1, 0), (3, 0), (3, 1), (2, 1), (2, -1), (1, 1), (3, -1)):
        plan.configure(mode)
        plan.set_parity(parity)
        out.zero_()
        plan.run(ws, out)
        plan.status()
        assert (to_host(out) == _of_class(values, parity)).all()
    plan.close()


# boards with 7 empty cells: a block each up to 4,999, packs from 5,000 on (the
# eight left over a block each)
@pytest.mark.parametrize("count, launches", [(16, 1), (600, 1), (4999, 1), (5000, 2 + 1)])
def test_boards_with_seven_empty_cells(count, launches):
    boards = inputs.midgame_boards(40, 7, 0xA44E)
    want = midgame_oracle(boards)
    at = np.arange(count) % 40
    assert (_run(boards[at], 7, 1, -1, launches) == want[at]).all()
    assert (_run(boards[at], 7, 1, 1, launches) == _of_class(want[at], 1)).all()


# 15 boards make no pack, 16 one, 17 one and a single board (too few fills to
# pay for both), 48 three
@pytest.mark.parametrize("count, launches", [(15, 2), (16, 2), (17, 2), (48, 2)])
@pytest.mark.parametrize("mode", [1, 2])
def test_around_the_pack_size(count, launches, mode):
    boards = inputs.midgame_boards(count, 8, 0xA44F)
    # the packs' roots are a launch of their own where a level is one
    level_launches = {15: 10, 16: 11, 17: 10, 48: 11}[count]
    assert (_run(boards, 8, mode, -1, launches if mode == 1 else level_launches) == midgame_oracle(boards)).all()


# a block each, of a warp up to 4 empty cells
@pytest.mark.parametrize("specs", [((3, 0),), ((5, 1),), ((40, 2),), ((9, 3), (2, 1)), ((70, 4),), ((7, 4), (3, 5))])
@pytest.mark.parametrize("parity", [-1, 0, 1])
def test_few_empty_cells(specs, parity):
    boards = _drawn(specs, 0xA450)
    kmax = max(k for _, k in specs)
    assert (_run(boards, kmax, 1, parity, 1) == _of_class(midgame_oracle(boards), parity)).all()
