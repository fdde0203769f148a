"""Root values of packed boards, read in the launch that wrote them: plans of
other boards of one shape run in turn in one workspace, so that a root read
before its level was done would be the other plan's.  Bit tables, compared
exactly."""
import pytest

from paper_1404_0743_gb300 import inputs
from tests.gpu_helpers import midgame_oracle, ready, to_host

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("parity", [-1, 1])
def test_each_run_reads_its_own_roots(parity):
    import torch
    pp = ready()
    count, k = 64, 8
    sets = [inputs.midgame_boards(count, k, 0x2007 + i) for i in range(2)]
    want = [midgame_oracle(b) for b in sets]
    if parity >= 0:
        from tests.test_gpu_parity import class_mask
        want = [w & class_mask(parity) for w in want]
    ws = torch.empty(pp.midgame_workspace_bytes(count, k), dtype=torch.uint8, device="cuda")
    plans = [pp.MidgamePlan(b, k) for b in sets]
    outs = [torch.zeros((count, 8), dtype=torch.int64, device="cuda") for _ in sets]
    for plan in plans:
        plan.configure(1)
        plan.set_parity(parity)
    for _ in range(8):
        for plan, out, values in zip(plans, outs, want):
            out.zero_()
            plan.run(ws, out)
            plan.status()
            assert (to_host(out) == values).all()
    for plan in plans:
        plan.close()
