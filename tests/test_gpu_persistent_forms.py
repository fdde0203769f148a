"""Single boards in the persistent launch: few fills go by lane pairs, many a
lane to a fill.  Either against the same boards a level at a time (which other
tests compare with the oracle).  Bit tables, compared exactly."""
import numpy as np
import pytest

from paper_1404_0743_gb300 import inputs
from tests.gpu_helpers import ready, to_host

pytestmark = pytest.mark.gpu


# 15 empty cells are 3.6 million fills: three boards are below the line, four
# above; one shape (a shared descriptor) and several
@pytest.mark.parametrize("deep", [3, 4])
@pytest.mark.parametrize("others", [(), (9, 9, 12, 8)])
def test_persistent_equals_levels(deep, others):
    import torch
    pp = ready()
    boards = np.concatenate([inputs.midgame_boards(deep, 15, 0xF0)] +
                            [inputs.midgame_boards(1, k, 0xF1 + i) for i, k in enumerate(others)])
    ws = torch.empty(pp.midgame_workspace_bytes(len(boards), 15), dtype=torch.uint8, device="cuda")
    got = []
    for mode in (2, 1):
        plan = pp.MidgamePlan(boards, 15)
        plan.configure(mode)
        out = torch.full((len(boards), 8), -1, dtype=torch.int64, device="cuda")
        ws.zero_()
        plan.run(ws, out)
        plan.status()
        got.append(to_host(out))
        plan.close()
    assert (got[0] == got[1]).all()
