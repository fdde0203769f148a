"""Midgame plans whose boards are solved sixteen to a pack: batches around the
pack size, several shapes mixed with boards left over, every launch mode and
parity class, against the oracle; larger shapes against the same boards in
batches too small for a pack.  Bit tables, compared exactly."""
import numpy as np
import pytest

from paper_1404_0743_gb300 import inputs
from tests.gpu_helpers import bits_to_bool, midgame_oracle, ready, to_host

pytestmark = pytest.mark.gpu


def _solve(pp, boards, kmax, mode=1, parity=-1):
    import torch
    plan = pp.MidgamePlan(boards, kmax)
    plan.set_parity(parity)
    plan.configure(mode)
    size = pp.midgame_workspace_bytes if parity < 0 else pp.midgame_parity_workspace_bytes
    ws = torch.empty(size(len(boards), kmax), dtype=torch.uint8, device="cuda")
    out = torch.full((len(boards), 8), -1, dtype=torch.int64, device="cuda")
    for _ in range(2):  # the second run finds the tables of the first
        plan.run(ws, out)
    plan.status()
    got = to_host(out)
    plan.close()
    return got


def _class_mask(parity):
    beta = np.arange(256)
    cls = (beta ^ beta >> 2 ^ beta >> 4 ^ beta >> 6) & 1
    return cls == parity


@pytest.fixture(scope="module")
def mixed():
    """17 boards with 6 empty cells (below the packs' least), 16 with 7, 35
    with 8 and 15 with 9 (no pack), shuffled, and their oracle values."""
    boards = np.concatenate([inputs.midgame_boards(n, k, 0x9ACC + 1000 * k)
                             for n, k in ((17, 6), (16, 7), (35, 8), (15, 9))])
    boards = boards[np.random.default_rng(5).permutation(len(boards))]
    return boards, midgame_oracle(boards)


@pytest.mark.parametrize("mode", [1, 2, 3])
@pytest.mark.parametrize("parity", [-1, 0, 1])
def test_mixed_batch(mixed, mode, parity):
    pp = ready()
    boards, want = mixed
    got = _solve(pp, boards, 9, mode, parity)
    if parity < 0:
        assert (got == want).all()
    else:
        keep = _class_mask(parity)
        assert (bits_to_bool(got) == (bits_to_bool(want) & keep)).all()


# 15 boards make no pack, 16 one, 17 one and a single board, 48 three
@pytest.mark.parametrize("count", [15, 16, 17, 48])
def test_around_the_pack_size(count):
    pp = ready()
    boards = inputs.midgame_boards(count, 7, 0x9ACC)
    assert (_solve(pp, boards, 7) == midgame_oracle(boards)).all()


@pytest.mark.parametrize("empties, parity", [(10, -1), (11, 1), (13, -1), (13, 0)])
def test_equals_boards_solved_one_by_one(empties, parity):
    pp = ready()
    boards = inputs.midgame_boards(32, empties, 0x9ACD)
    want = np.concatenate([_solve(pp, boards[i:i + 8], empties, 2, parity) for i in range(0, 32, 8)])
    for mode in (1, 2):
        assert (_solve(pp, boards, empties, mode, parity) == want).all()
