"""The host-resident loop: the buffers it takes and the plans it refuses."""
import pytest
import torch

from paper_1808_02638_gb300 import claw, inputs
from paper_1808_02638_gb300.solver import Hierarchy

pytestmark = pytest.mark.gpu


def _hierarchy(n, patch):
    run = inputs.config1(n, patch)
    H = Hierarchy([run], [[inputs.init_q(run, run.levels[0])]], rho0=1.0, K0=4.0)
    H.init_dt()
    H.fused = True
    return H


def test_pieces_behind_the_packed_interiors_are_refused():
    H = _hierarchy(64, 32)
    host = H.pack().cpu().pin_memory()
    n = host.numel()
    stage = [torch.empty(n, dtype=torch.float64, device="cuda") for _ in range(2)]
    before = H.q[0][0].clone()
    for ranges in ([(0, n + 1)], [(n, n + 8)], [(0, 1 << 40)], [(1 << 40, 1 << 41)]):
        with pytest.raises(claw.ClawError) as e:
            claw.claw_steps_from_host(H.ctx, H.q[0][0], H.q[0][1], None, H.dt, H.smax, host,
                                      torch.empty_like(host).pin_memory(), *stage, 1, [(0, 4)], ranges, [[0]])
        assert e.value.status == claw.CLAW_EINVAL
    torch.cuda.synchronize()
    assert torch.equal(H.q[0][0], before)
    H.close()
