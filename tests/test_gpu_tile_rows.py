"""Levels of few tiles, whose tiles are lower than the kernel's: every cell is stepped exactly once and
to the same bits whatever the tile shape, for the two kernels that lower them."""
import numpy as np
import pytest

from paper_1808_02638_gb300 import claw, inputs, tune
from paper_1808_02638_gb300.solver import Hierarchy

pytestmark = pytest.mark.gpu

BOXES = {"thin": [(0, 0, 4, 61)], "flat": [(0, 0, 130, 5)], "odd": [(0, 0, 33, 47)], "wide": [(0, 0, 190, 170)],
         "even": [(0, 0, 256, 256)], "mixed": [(0, 0, 40, 64), (40, 0, 24, 20), (40, 20, 24, 44), (64, 0, 8, 64)]}


@pytest.mark.parametrize("system", ["cellwise", "swe"])
@pytest.mark.parametrize("boxes", sorted(BOXES))
def test_the_step_does_not_depend_on_the_tile_shape(boxes, system):
    bx = BOXES[boxes]
    nx, ny = max(b[0] + b[2] for b in bx), max(b[1] + b[3] for b in bx)
    run = inputs.Run(0.0, 0.0, nx * 0.02, ny * 0.02, limiter=4)
    run.levels = [inputs.Level(nx, ny, 0.02, 0.02, bx)]
    lev = run.levels[0]
    rng = np.random.default_rng(5)
    pool = rng.uniform(0.7, 1.4, lev.qsize)
    if system == "swe":
        H = Hierarchy([run], [[pool]], system="shallow_water", grav=1.0)
    else:
        H = Hierarchy([run], [[pool]], [[rng.uniform(0.5, 2.0, lev.csize)]], [[rng.uniform(0.5, 2.0, lev.csize)]])
    H.dt.fill_(0.9 * 0.02 / 6.0)
    claw.claw_fill_ghost(H.ctx, 0, H.q[0][0], None, None, 0.0)
    got = []
    for tiling in tune.candidates_for(H):
        try:
            claw.claw_set_tiling(H.ctx, 0, *tiling)
        except claw.ClawError:
            continue   # bulk copies need an even width
        H.q[0][1].fill_(float("nan"))
        claw.claw_level_step(H.ctx, 0, H.q[0][0], H.q[0][1], H.aux[0], H.dt, H.smax)
        assert H.sync_status() == claw.CLAW_OK
        got.append([H.interior(0, 0, b, pool=H.q[0][1]) for b in range(len(bx))])
    assert len(got) >= 2
    for b in range(len(bx)):
        assert np.isfinite(got[0][b]).all()
        for other in got[1:]:
            np.testing.assert_array_equal(other[b], got[0][b])
    H.close()
