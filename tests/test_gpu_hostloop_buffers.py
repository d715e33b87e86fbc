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


def _after(n, patch, nsteps):
    H = _hierarchy(n, patch)
    for _ in range(nsteps):
        H.coarse_step()
    out, dt = H.pack().cpu(), float(H.dt[0])
    H.close()
    return out, dt


@pytest.mark.parametrize("nsteps", [1, 3, 4])
@pytest.mark.parametrize("kind", ["device", "longer", "longer strided", "read only", "two rows"])
def test_every_kind_of_buffer_that_copies_is_taken(kind, nsteps):
    n, patch = 64, 16
    want, dt = _after(n, patch, nsteps)
    before, _ = _after(n, patch, nsteps - 1)
    H = _hierarchy(n, patch)
    host = H.pack().cpu()
    m = host.numel()
    a, b = host.clone(), torch.empty_like(host)
    if kind == "device":
        a, b = a.cuda(), b.cuda()
    elif kind == "longer":
        b = torch.full((m + 7,), -1.0, dtype=torch.float64).pin_memory()
    elif kind == "longer strided":
        b = torch.full((2 * (m + 7),), -1.0, dtype=torch.float64)[::2]
    elif kind == "two rows":
        a, b = a.view(2, -1), torch.empty(2, m, dtype=torch.float64)[:, ::2]
    elif kind == "read only":   # one step reads host_a and writes host_b alone
        if nsteps > 1:
            pytest.skip("the second step writes host_a")
        a = a.requires_grad_(True)
        b = torch.empty(2 * m, dtype=torch.float64)[::2]
    out = H.steps_from_host(a, b, nsteps)
    torch.cuda.synchronize()
    assert out is (b if nsteps % 2 else a)
    last, other = (b, a) if nsteps % 2 else (a, b)
    assert torch.equal(last.detach().cpu().reshape(-1)[:m], want)
    assert torch.equal(other.detach().cpu().reshape(-1)[:m], before)
    if kind.startswith("longer"):
        assert bool((b[m:] == -1.0).all())
    assert float(H.dt[0]) == dt and H.sync_status() == 0
    H.close()


def test_no_steps_leave_everything_as_it_is():
    H = _hierarchy(64, 32)
    host = H.pack().cpu()
    a, b = host.clone(), torch.zeros_like(host)
    for nsteps in (0, -1):
        assert H.steps_from_host(a, b, nsteps) is a
    assert torch.equal(a, host) and not bool(b.any())
    with pytest.raises(ValueError):
        H.steps_from_host(a, b[:-1], 1)
    with pytest.raises(ValueError):
        H.steps_from_host(a[:-1], b, 1)
    H.close()


@pytest.mark.parametrize("nsteps", [1, 2])
def test_single_precision_buffers_hold_the_rounded_states(nsteps):
    n, patch = 64, 16
    H = _hierarchy(n, patch)
    host = H.pack().cpu()
    a, b = host.float(), torch.empty(host.numel())
    D = _hierarchy(n, patch)   # the same steps of the state that the buffer holds
    x, y = a.double().pin_memory(), torch.empty_like(host).pin_memory()
    want = D.steps_from_host(x, y, nsteps)
    out = H.steps_from_host(a, b, nsteps)
    torch.cuda.synchronize()
    assert torch.equal(out, want.float()) and float(H.dt[0]) == float(D.dt[0])
    H.close()
    D.close()
