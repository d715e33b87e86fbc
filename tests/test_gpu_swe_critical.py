"""The shallow-water step where flows turn supercritical: edges on either side of |u| = c in either
direction, at rest, and mixed within a tile, against the oracle's step."""
import numpy as np
import pytest

import oracle
from paper_1808_02638_gb300 import claw, inputs
from paper_1808_02638_gb300.solver import Hierarchy

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("order,transverse", [(2, 2), (2, 1), (2, 0), (1, 1)])
@pytest.mark.parametrize("u0,v0", [(0.0, 0.0), (0.9, -0.2), (-1.6, 0.3), (0.2, 1.5), (-2.5, -2.5), (1.0, 0.0)])
def test_sub_and_supercritical_edges_match_the_oracle(u0, v0, order, transverse):
    # 30 roundings of 2^-53 of the largest value of the update's terms (speeds below 6, CFL below 1)
    nx, ny = 37, 45
    rng = np.random.default_rng(11)
    q = np.empty((3, ny + 4, nx + 4))
    q[0] = rng.uniform(0.6, 1.6, q[0].shape)
    # a band across the grid flows twice as fast: both kinds of edges in one tile
    speed = np.where(np.arange(nx + 4)[None, :] % 20 < 10, 1.0, 2.0)
    q[1], q[2] = q[0] * u0 * speed, q[0] * v0 * speed
    for limiter in (1, 2, 3, 4):
        run = inputs.Run(0.0, 0.0, nx * 0.02, ny * 0.02, limiter=limiter, order=order, transverse=transverse)
        run.levels = [inputs.Level(nx, ny, 0.02, 0.02, [(0, 0, nx, ny)])]
        pool = np.zeros(run.levels[0].qsize)
        inputs.box_view(pool, 0, nx, ny, 3)[...] = q
        H = Hierarchy([run], [[pool]], system="shallow_water", grav=1.0)
        H.dt.fill_(0.9 * 0.02 / 8.0)
        claw.claw_level_step(H.ctx, 0, H.q[0][0], H.q[0][1], None, H.dt, H.smax)
        got = H.interior(0, 0, 0, pool=H.q[0][1])
        want = oracle.swe_step(q, 0.02, 0.02, 0.9 * 0.02 / 8.0, order=order, transverse=transverse, limiter=limiter, grav=1.0)
        want = (want[0] if isinstance(want, tuple) else want)[:, 2:-2, 2:-2]
        assert np.abs(got - want).max() <= 30 * 2.0 ** -53 * 6.0 * np.abs(q).max()
        assert H.sync_status() == claw.CLAW_OK
        H.close()
