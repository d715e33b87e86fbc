"""Launches that carry the work of several: the level-step with the conservation fix's edges beside its
tiles, the average with the fix's corrections, and the fill of both kinds of ghosts give what the
separate entry points give, bit for bit; averages for every kind of ratio equal numpy's."""
import numpy as np
import pytest
import torch

from paper_1808_02638_gb300 import claw, inputs
from paper_1808_02638_gb300.solver import Hierarchy

pytestmark = pytest.mark.gpu


def _hierarchy(system, ratio, limiter, order=2, transverse=2):
    run = inputs.Run(*inputs.PULSE_DOMAIN, limiter=limiter, order=order, transverse=transverse, bc=(1, 1, 2, 2))
    run.levels = inputs.amr_levels(run, 48, ratio, [(0.2, 0.45), (0.25, 0.35)], [2002, 2003])
    swe = system == "shallow_water"
    q0 = [inputs.init_swe(run, lev, u0=0.3, v0=-0.2) if swe else inputs.init_q(run, lev) for lev in run.levels]
    H = Hierarchy([run], [q0], reflux=True, system=system, rho0=1.0, K0=4.0, grav=1.0)
    H.init_dt()
    H.coarse_step()
    return H


@pytest.mark.parametrize("limiter", range(5))
@pytest.mark.parametrize("system,ratio", [("acoustics", 2), ("acoustics", 4), ("shallow_water", 2)])
@pytest.mark.parametrize("order,transverse", [(2, 2), (2, 0), (1, 1)])
def test_step_with_the_fix_s_edges_equals_separate_launches(system, ratio, limiter, order, transverse):
    H = _hierarchy(system, ratio, limiter, order, transverse)
    q = [H.q[L][H.cur[L]] for L in range(3)]
    claw.claw_fill_ghost(H.ctx, 0, q[0])
    for L in (1, 2):
        claw.claw_fill_ghost(H.ctx, L, q[L], q[L - 1], q[L - 1], 0.5)
    for L in range(3):
        out = []
        for merged in (False, True):
            new, smax = torch.zeros_like(q[L]), torch.zeros_like(H.smax)
            fine = torch.full_like(H.rbuf[L], 0.25) if L else None
            coarse = torch.full_like(H.rbuf[L + 1], 7.0) if L < 2 else None
            if merged:
                claw.claw_level_step_reflux(H.ctx, L, q[L], new, H.dt, smax, q[L - 1] if L else None, fine, coarse)
            else:
                if L:
                    claw.claw_reflux_fine(H.ctx, L, q[L], q[L - 1], H.dt, fine)
                if L < 2:
                    claw.claw_reflux_coarse(H.ctx, L + 1, q[L], H.dt, coarse)
                claw.claw_level_step(H.ctx, L, q[L], new, None, H.dt, smax)
            out.append((new, smax, fine, coarse))
        for a, b in zip(*out):
            assert (a is None and b is None) or torch.equal(a, b)
        assert L == 2 or not torch.equal(out[0][3], torch.full_like(out[0][3], 7.0))
    for L in (1, 2):
        a, b = q[L - 1].clone(), q[L - 1].clone()
        buf = torch.rand_like(H.rbuf[L])
        claw.claw_average_down(H.ctx, L, q[L], a)
        claw.claw_reflux_apply(H.ctx, L, buf, H.dt, a)
        claw.claw_average_down_reflux(H.ctx, L, q[L], b, buf, H.dt)
        assert torch.equal(a, b)
    assert H.sync_status() == claw.CLAW_OK


def test_merged_calls_refuse_what_the_separate_ones_do():
    H = _hierarchy("acoustics", 2, 4)
    q, new = H.q[0]
    for args in ((0, q, new, H.dt, H.smax, q, H.rbuf[1], None), (1, H.q[1][0], H.q[1][1], H.dt, H.smax, None, H.rbuf[1], None),
                 (2, H.q[2][0], H.q[2][1], H.dt, H.smax, H.q[1][0], None, H.rbuf[1]), (0, q, q, H.dt, H.smax, None, None, None)):
        with pytest.raises(claw.ClawError) as e:
            claw.claw_level_step_reflux(H.ctx, *args)
        assert e.value.status == claw.CLAW_EINVAL
    with pytest.raises(claw.ClawError):
        claw.claw_average_down_reflux(H.ctx, 1, H.q[1][0], q, None, H.dt)


@pytest.mark.parametrize("ratio", [2, 3, 4, 5])
def test_averages_of_every_ratio(ratio):
    run = inputs.Run(*inputs.PULSE_DOMAIN)
    n = 40
    boxes = [(0, 0, 2 * ratio, 2 * ratio), (4 * ratio, 6 * ratio, 30 * ratio, 17 * ratio)]
    run.levels = [inputs.Level(n, n, 2 / n, 2 / n, [(0, 0, n, n)]),
                  inputs.Level(n * ratio, n * ratio, 2 / n / ratio, 2 / n / ratio, boxes, ratio)]
    H = Hierarchy([run], [[inputs.init_q(run, lev) for lev in run.levels]], rho0=1.0, K0=4.0)
    qf = torch.rand_like(H.q[1][0])
    qc = torch.rand_like(H.q[0][0])
    want = inputs.box_view(qc.cpu().numpy().copy(), 0, n, n, 3)
    claw.claw_average_down(H.ctx, 1, qf, qc)
    lev, f = run.levels[1], qf.cpu().numpy()
    for k, (i, j, nx, ny) in enumerate(lev.boxes.tolist()):
        v = inputs.box_view(f, lev.qoff[k], nx, ny, 3)[:, 2:-2, 2:-2].reshape(3, ny // ratio, ratio, nx // ratio, ratio)
        s = np.zeros(v.shape[:2] + v.shape[3:4])
        for b in range(ratio):
            for a in range(ratio):
                s = s + v[:, :, b, :, a]
        ci, cj = i // ratio + 2, j // ratio + 2
        want[:, cj:cj + ny // ratio, ci:ci + nx // ratio] = s / ratio ** 2
    assert np.array_equal(inputs.box_view(qc.cpu().numpy(), 0, n, n, 3), want)
