"""Which tiles the uniform-medium step takes in fixed point, and how exact either path is: against the
same step in extended precision, by component, with small states beside a large jump."""
import numpy as np
import pytest

from paper_1808_02638_gb300 import claw, inputs
from paper_1808_02638_gb300.solver import Hierarchy

LD = np.longdouble
pytestmark = [pytest.mark.gpu, pytest.mark.skipif(np.finfo(LD).nmant < 63, reason="no extended precision")]

Z, C = 1.7, 1.7   # rho = 1, K = Z Z
ROUNDING = 2.0 ** -53


def _step(q, nu, h, order, transverse, limiter, tiling):
    """(3, ny, nx) after a step of the (3, ny + 4, nx + 4) state q"""
    ny, nx = q.shape[1] - 4, q.shape[2] - 4
    run = inputs.Run(0.0, 0.0, nx * h, ny * h, limiter=limiter, order=order, transverse=transverse)
    run.levels = [inputs.Level(nx, ny, h, h, [(0, 0, nx, ny)])]
    pool = np.zeros(run.levels[0].qsize)
    inputs.box_view(pool, 0, nx, ny, 3)[...] = q
    H = Hierarchy([run], [[pool]], rho0=1.0, K0=Z * Z, tiling=tiling)
    dt = nu * h / C
    H.dt.fill_(dt)
    claw.claw_level_step(H.ctx, 0, H.q[0][0], H.q[0][1], None, H.dt, H.smax)
    out = H.interior(0, 0, 0, pool=H.q[0][1])
    assert H.sync_status() == claw.CLAW_OK
    H.close()
    return out, LD(dt) * LD(1.0 / h) * LD(C)


def _sweep(p, u, nu, second):
    """twice the x-updates of p / Z and u over -nu, and twice the x-fluctuation pressure / Z into a cell, all rows"""
    dp, du = np.diff(p, axis=1) / LD(Z), np.diff(u, axis=1)
    a1, a2 = du - dp, du + dp

    def mc(a, b):   # phi(b / a) a
        s = np.where(a < 0, LD(-1), LD(1))
        x, y = s * a, s * b
        return s * np.where((x > 0) & (y > 0), np.minimum((x + y) / 2, 2 * np.minimum(x, y)), LD(0))

    m1, m2 = mc(a1[:, 1:-1], a1[:, 2:]), mc(a2[:, 1:-1], a2[:, :-2])
    k = (1 - nu) if second else LD(0)
    bp, bu = k * np.diff(m2 - m1, axis=1), k * np.diff(m1 + m2, axis=1)
    ap, au = a2[:, 1:-2] + a1[:, 2:-1], a2[:, 1:-2] - a1[:, 2:-1]
    return ap + bp / 2, au + bu / 2, ap + bp


def _want(q, nu, order, transverse):
    """the step in extended precision, dx = dy, MC; full transverse corrections or none"""
    p, u, v = q.astype(LD)
    X, U, D = _sweep(p, u, nu, order == 2)
    Y, V, E = (t.T for t in _sweep(p.T, v.T, nu, order == 2))
    i = slice(2, -2)
    P, U, V = p[i, i] / LD(Z) - nu / 2 * (X[i] + Y[:, i]), u[i, i] - nu / 2 * U[i], v[i, i] - nu / 2 * V[:, i]
    if transverse:
        D, E = D[1:-1], E[:, 1:-1]
        P = P - nu * nu / 8 * (D[2:] + D[:-2] - 2 * D[1:-1] + E[:, 2:] + E[:, :-2] - 2 * E[:, 1:-1])
        U = U + nu * nu / 8 * (E[:, 2:] - E[:, :-2])
        V = V + nu * nu / 8 * (D[2:] - D[:-2])
    return np.stack([P * LD(Z), U, V])


def _grid(nx, ny):
    return np.linspace(-1.0, 1.0, nx + 4)[None, :], np.linspace(-1.0, 1.0, ny + 4)[:, None]


@pytest.mark.parametrize("tiling", [(32, 32, 1, 256), (32, 16, 0, 256), (16, 16, 1, 192)])
def test_each_component_errs_by_its_own_rounding_where_jumps_are_moderate(tiling):
    # One fused multiply-add forms each component: half a unit in the last place, at most 2^-53 of the value, and
    # 5 units of 2^(e - 58), here below 2^-5 of that.  The FP64 phases form p by five of them (3 roundings and
    # more), so this also says that the tiles go the other way.
    x, y = _grid(64, 48)
    w = [np.cos(5.1 * x + 3.3 * y + k) for k in range(3)]
    q = np.stack([1.0 + 0.3 * w[0], 0.2 * w[1], 0.1 * w[2]])
    got, nu = _step(q, 0.9, 0.02, 2, 2, 4, tiling)
    err = np.abs(got - _want(q, nu, 2, 2)).max(axis=(1, 2)).astype(float)
    assert np.all(err <= 1.2 * ROUNDING * np.abs(q).max(axis=(1, 2))), err / ROUNDING


def _beside_jumps(ratio, n=128):
    """a state of about 2 ratio in wave units in every component, with a jump of 0.9 Z in p in every 32 x 32
    cells: |dp| / Z < 2^e with e = 1 (as the exponents of dp and Z bound it)"""
    rng = np.random.default_rng(int(1e6 * ratio))
    q = 2.0 * ratio * (1.0 + 1.0e-3 * rng.uniform(-1.0, 1.0, (3, n + 4, n + 4)))
    q[0] *= Z
    q[0, 8:-2:32, 8:-2:32] += 0.9 * Z
    far = np.ones((n, n), dtype=bool)
    for j in range(6, n, 32):
        for i in range(6, n, 32):
            far[j - 3:j + 4, i - 3:i + 4] = False
    return q, far


@pytest.mark.parametrize("order,transverse", [(1, 0), (2, 2)])
@pytest.mark.parametrize("ratio", [0.6, 0.27, 0.2, 0.14, 0.07, 0.03, 2.0 ** -10, 2.0 ** -30, 2.0 ** -52])
def test_small_states_beside_a_large_jump_keep_their_precision(ratio, order, transverse):
    # Cells out of the jumps' reach, relative to their own state.  The FP64 phases: 2^-53 a fused multiply-add, of
    # which the first-order step without transverse terms has two for p and one for u and v, the full step
    # five and three.  Beside it, with jumps of up to 2e-3 of the state (twice that for a strength): the new state
    # is larger by up to 0.002; two strengths, rounded, and their sum or difference, nu / 2 (2 x 0.004 + 0.008);
    # the coefficients' roundings, 4 x 0.002: 0.02 in all, and three times that with the limited and the
    # transverse terms.  Fixed point: 2^-53 for its one multiply-add, and 5 units of 2^(e - 58), where it is taken:
    # from 2^(e - 2) and 2^(e - 4) on.
    q, far = _beside_jumps(ratio)
    for nu in (0.9, 0.55):
        got, nu_ = _step(q, nu, 0.02, order, transverse, 4, (32, 32, 1, 256))
        rel = np.abs(got - _want(q, nu_, order, transverse)) / np.abs(q[:, 2:-2, 2:-2])
        rel = rel[:, far].max(axis=1).astype(float) / ROUNDING
        if ratio >= (0.25 if order == 1 else 0.0625):
            bound = np.full(3, 1.02 + 5 * 2.0 ** -5 / ratio)
        else:
            bound = np.array([2.02, 1.02, 1.02] if order == 1 else [5.06, 3.06, 3.06])
        assert np.all(rel <= bound), (rel, bound)


@pytest.mark.parametrize("tiling", [(32, 32, 1, 256), (32, 32, 0, 512), (32, 16, 2, 256), (16, 16, 1, 128), (16, 16, 0, 192)])
def test_a_state_without_jumps_comes_out_as_it_is(tiling):
    # bit for bit, signs of zeros included, whatever its size
    for state in ((0.0, 0.0, 0.0), (0.0, -0.0, 0.0), (-0.0, 0.0, -0.0), (5.0e-324, 0.0, 0.0), (1.0e-310, -1.0e-312, 3.0e-320),
                  (1.0e-290, 0.0, -1.0e-300), (1.0, -0.0, 1.0e-300), (1.0e300, 1.0e290, 0.0)):
        q = np.broadcast_to(np.array(state)[:, None, None], (3, 52, 70)).copy()
        got, _ = _step(q, 0.9, 0.02, 2, 2, 4, tiling)
        assert np.array_equal(got.view(np.int64), q[:, 2:-2, 2:-2].copy().view(np.int64))


def test_the_smallest_jumps_are_not_taken_for_none():
    # subnormal jumps, whose upper words are zero, on zeros: some of it moves on, as the exact step has it within a
    # unit of the smallest subnormal for each of the FP64 phases' operations (24 for all terms of p)
    for size in (2.0 ** -1043, 2.0 ** -1060):
        q = np.zeros((3, 52, 52))
        q[0, 24:28, 24:28] = size
        got, nu = _step(q, 0.9, 0.02, 2, 2, 4, (32, 32, 1, 256))
        want = _want(q, nu, 2, 2)
        assert np.abs(got - want).max() <= 24 * 2.0 ** -1074
        assert np.count_nonzero(got[1]) > 8 and np.abs(got[1]).max() > size / 8
        assert not got[:, :16, :16].any()
