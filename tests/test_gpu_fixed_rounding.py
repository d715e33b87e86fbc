"""The rounding of the uniform-medium step's fixed-point tiles has no preferred direction: totals are
conserved as well as in FP64, and what is symmetric stays symmetric bit for bit."""
import math

import numpy as np
import pytest
import torch

from paper_1808_02638_gb300 import inputs
from paper_1808_02638_gb300.solver import Hierarchy

pytestmark = pytest.mark.gpu

PERIODIC, WALL = 1, 2


def _hierarchy(q, dx, dy, bc, limiter, order, transverse, tiling, cfl=0.9):
    ny, nx = q.shape[1:]
    run = inputs.Run(0.0, 0.0, nx * dx, ny * dy, bc=(bc,) * 4, cfl=cfl, limiter=limiter, order=order, transverse=transverse)
    run.levels = [inputs.Level(nx, ny, dx, dy, [(0, 0, nx, ny)])]
    pool = np.zeros(run.levels[0].qsize)
    inputs.box_view(pool, 0, nx, ny, 3)[:, 2:-2, 2:-2] = q
    H = Hierarchy([run], [[pool]], rho0=1.0, K0=2.89, tiling=tiling)
    H.init_dt()
    H.fused = True
    return H


def _run(H, n):
    for _ in range(n):
        H.coarse_step()
    torch.cuda.synchronize()
    assert H.sync_status() == 0
    return H.interior(0, 0, 0)


def _symmetric_ring(n):
    c = (np.arange(n) + 0.5) * (2.0 / n) - 1.0
    r = np.sqrt(c[None, :] ** 2 + c[:, None] ** 2)
    p = 1.0 + 0.4 * np.exp(-((r - 0.4) / 0.15) ** 2)
    p = p[:, ::-1] + p
    p = 0.25 * (p + p[::-1])
    return np.stack([p, np.zeros_like(p), np.zeros_like(p)])


@pytest.mark.parametrize("tiling", [(32, 32, 1, 256), (32, 16, 0, 256), (16, 16, 1, 192)])
@pytest.mark.parametrize("limiter", [0, 1, 2, 3, 4])
def test_a_mirror_symmetric_state_stays_so_bit_for_bit(tiling, limiter):
    n = 64
    for dy, order, transverse in ((2.0 / n, 2, 2), (3.0 / n, 2, 2), (1.5 / n, 2, 1), (2.0 / n, 1, 1)):
        H = _hierarchy(_symmetric_ring(n), 2.0 / n, dy, WALL, limiter, order, transverse, tiling,
                       cfl=0.9 if transverse else 0.4)
        q = _run(H, 30)
        H.close()
        p, u, v = q
        assert np.array_equal(p, p[:, ::-1]) and np.array_equal(p, p[::-1])
        assert np.array_equal(u, -u[:, ::-1]) and np.array_equal(u, u[::-1])
        assert np.array_equal(v, v[:, ::-1]) and np.array_equal(v, -v[::-1])
        assert np.abs(u).max() > 0.01 and np.abs(v).max() > 0.01


@pytest.mark.parametrize("limiter", [1, 2, 3, 4])
def test_a_state_of_the_other_sign_gives_the_other_sign(limiter):
    rng = np.random.default_rng(limiter)
    q = rng.uniform(-1.0, 1.0, (3, 49, 70)) + np.array([3.0, 1.0, 1.0])[:, None, None]
    a, b = (_run(_hierarchy(s * q, 0.02, 0.03, PERIODIC, limiter, 2, 2, (32, 32, 1, 256)), 5) for s in (1.0, -1.0))
    assert np.array_equal(a, -b)


@pytest.mark.parametrize("kind", ["ring", "sawtooth"])
@pytest.mark.parametrize("ratio", [1.0, 1.6])
@pytest.mark.parametrize("limiter", [3, 4])
def test_totals_wander_but_do_not_drift(kind, ratio, limiter):
    # One rounding of p to 2^-53 of a value below 2 errs by 0.29 units of 2^-52 rms, so n steps of N cells
    # move the total by 0.29 2^-52 sqrt(n N) rms.  Six times that, for the last rounding alone; errors of a
    # preferred sign grow with n instead (rounding downwards: 5 to 8e-12 here).  The totals of u and v
    # likewise, for values below 1/2.
    n, steps = 64, 1000
    x = ((np.arange(n) + 0.5) / n)[None, :]
    y = ((np.arange(n) + 0.5) / n)[:, None]
    if kind == "ring":
        q = _symmetric_ring(n)
    else:
        q = np.stack([1.0 + 0.3 * ((4 * x + 3 * y) % 1), 0.1 + 0.1 * ((3 * x + 2 * y) % 1), -0.2 + 0.1 * ((x + 5 * y) % 1)])
    H = _hierarchy(q, 2.0 / n, ratio * 2.0 / n, PERIODIC, limiter, 2, 2, (32, 32, 1, 256))
    out = _run(H, steps)
    H.close()
    move = np.abs([math.fsum(o.ravel().tolist() + (-i).ravel().tolist()) for o, i in zip(out, q)])
    bound = 6 * 0.29 * 2.0 ** -52 * np.sqrt(steps * n * n)
    assert move[0] <= bound and np.all(move[1:] <= 0.25 * bound), (move, bound)

