"""The host-resident loop at the sizes where its number of pieces changes, for buffers it copies
through, and its argument checks: the states equal those of device-resident steps bit for bit."""
import numpy as np
import pytest
import torch

from paper_1808_02638_gb300 import claw, inputs
from paper_1808_02638_gb300.solver import Hierarchy

pytestmark = pytest.mark.gpu


def _pair(n, patch):
    run = inputs.config1(n, patch)
    q = inputs.init_q(run, run.levels[0])
    out = []
    for _ in range(2):
        H = Hierarchy([run], [[q]], rho0=1.0, K0=4.0)
        H.init_dt()
        H.fused = True
        out.append(H)
    return out


@pytest.mark.parametrize("n,patch,nsteps", [(32, 32, 1), (64, 16, 4), (352, 32, 3), (384, 32, 2)])
@pytest.mark.parametrize("kind", ["pinned", "pageable", "strided", "float32"])
def test_packed_and_pool_states_equal_device_steps(n, patch, nsteps, kind):
    A, B = _pair(n, patch)
    for _ in range(nsteps):
        A.coarse_step()
    host = B.pack().cpu()
    if kind == "pinned":
        a, b = host.pin_memory(), torch.empty_like(host).pin_memory()
    elif kind == "pageable":
        a, b = host, torch.empty_like(host)
    elif kind == "strided":
        a, b = (torch.empty(2 * host.numel(), dtype=torch.float64)[::2] for _ in range(2))
        a.copy_(host)
    else:   # the state rounds to what the buffer holds when it is copied out
        a, b = host.float(), torch.empty_like(host).float()
        assert torch.equal(a.double(), host) or kind == "float32"
    out = B.steps_from_host(a, b, nsteps)
    torch.cuda.synchronize()
    assert out is (b if nsteps % 2 else a)
    want = A.pack().cpu()
    if kind == "float32":
        assert np.abs(out.double() - want).max() < 1e-5
    else:
        assert torch.equal(out.contiguous(), want)
        assert float(A.dt[0]) == float(B.dt[0])
    assert B.sync_status() == 0


def test_invalid_plans_are_refused():
    _, B = _pair(64, 32)
    host = B.pack().cpu().pin_memory()
    args = [B.ctx, B.q[0][0], B.q[0][1], None, B.dt, B.smax, host, torch.empty_like(host).pin_memory(),
            torch.empty(host.numel(), dtype=torch.float64, device="cuda"),
            torch.empty(host.numel(), dtype=torch.float64, device="cuda"), 1]
    whole = (0, host.numel())
    for pieces, ranges, needs in (([(0, 5)], [whole], [[0]]), ([(0, 4)], [(-1, 4)], [[0]]), ([(0, 4)], [(8, 4)], [[0]]),
                                  ([(0, 4)], [whole], [[1]]), ([(3, 2)], [whole], [[0]])):
        with pytest.raises(claw.ClawError) as e:
            claw.claw_steps_from_host(*args, pieces, ranges, needs)
        assert e.value.status == claw.CLAW_EINVAL
    with pytest.raises(claw.ClawError):
        claw.claw_steps_from_host(*args[:-2], None, 1, [(0, 4)], [whole], [[0]])
