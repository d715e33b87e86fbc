"""The uniform-medium step's fixed-point tiles and the FP64 phases that take the tiles those leave
over: one step against the oracle at tile edges and remainders, and over states that choose either
path (backgrounds, exponents, media, CFL numbers above 1, non-finite values)."""
import numpy as np
import pytest

import oracle
from paper_1808_02638_gb300 import claw, inputs
from paper_1808_02638_gb300.solver import Hierarchy

pytestmark = pytest.mark.gpu

TILINGS = [(32, 32, 1, 256), (32, 32, 2, 256), (32, 32, 0, 512), (32, 16, 2, 256), (32, 16, 1, 256), (16, 16, 1, 128)]
# per value about 25 roundings of at most 2^-53 of the largest value of the state in wave units
# (p, Z u, Z v), on either side
TOL = 50 * 2.0 ** -53


def _field(kind, nx, ny, rng):
    x = np.linspace(-1.0, 1.0, nx + 4)[None, :]
    y = np.linspace(-1.0, 1.0, ny + 4)[:, None]
    r2 = (x - 0.1) ** 2 + (y + 0.2) ** 2
    waves = [np.cos(5.1 * x + 3.3 * y + k) for k in range(3)]
    if kind == "background":      # small waves on a large pressure
        return np.stack([1.0e5 + waves[0], 2.0e-3 * waves[1], 1.0e-3 * waves[2]])
    if kind == "zero":            # decaying fronts on a zero background
        return np.stack([np.exp(-60.0 * r2), 0.3 * np.exp(-80.0 * r2) * x, 0.0 * r2])
    if kind == "rest":            # a constant state with one disturbed cell
        q = np.zeros((3, ny + 4, nx + 4)) + np.array([1.5, 0.25, -0.125])[:, None, None]
        q[0, ny // 2, nx // 2] += 1.0e-6
        return q
    if kind == "noise":
        return rng.uniform(-1.0, 1.0, (3, ny + 4, nx + 4)) + np.array([2.0, 0.0, 0.0])[:, None, None]
    scale = {"tiny": 1.0e-120, "large": 1.0e120}.get(kind, 1.0)
    return scale * np.stack([1.0 + 0.3 * waves[0], 0.2 * waves[1], 0.1 * waves[2]])


def _step(q, dx, dy, dt, limiter, order, transverse, rho0, K0, tiling):
    ny, nx = q.shape[1] - 4, q.shape[2] - 4
    run = inputs.Run(0.0, 0.0, nx * dx, ny * dy, limiter=limiter, order=order, transverse=transverse)
    run.levels = [inputs.Level(nx, ny, dx, dy, [(0, 0, nx, ny)])]
    pool = np.zeros(run.levels[0].qsize)
    inputs.box_view(pool, 0, nx, ny, 3)[...] = q
    if nx % 2:
        tiling = (tiling[0], tiling[1], 0, tiling[3])
    H = Hierarchy([run], [[pool]], rho0=rho0, K0=K0, tiling=tiling)
    H.dt.fill_(dt)
    claw.claw_level_step(H.ctx, 0, H.q[0][0], H.q[0][1], None, H.dt, H.smax)
    out = H.interior(0, 0, 0, pool=H.q[0][1])
    status = H.sync_status()
    H.close()
    return out, status


def _check(q, dx, dy, dt, limiter, order, transverse, rho0, K0, tiling):
    ones = np.ones(q.shape[1:])
    want = oracle.step(q, rho0 * ones, K0 * ones, dx, dy, dt, order=order, transverse=transverse, limiter=limiter)
    want = (want[0] if isinstance(want, tuple) else want)[:, 2:-2, 2:-2]
    got, status = _step(q, dx, dy, dt, limiter, order, transverse, rho0, K0, tiling)
    Z = np.sqrt(rho0 * K0)
    s = max(np.abs(q[0]).max(), Z * np.abs(q[1:]).max())
    err = np.abs(got - want).max(axis=(1, 2)) * np.array([1.0, Z, Z])
    assert status == claw.CLAW_OK and np.all(err <= TOL * s), err / s


@pytest.mark.parametrize("limiter", range(5))
@pytest.mark.parametrize("tiling", TILINGS)
def test_tile_edges_and_remainders(tiling, limiter):
    rng = np.random.default_rng(limiter)
    for nx, ny in ((1, 1), (2, 3), (15, 17), (33, 31), (36, 49), (66, 70)):
        for order, transverse in ((2, 2), (2, 1), (2, 0), (1, 1), (1, 0)):
            q = _field("noise", nx, ny, rng)
            _check(q, 0.02, 0.03, 0.4 * 0.02 / 2.0, limiter, order, transverse, 1.0, 4.0, tiling)


@pytest.mark.parametrize("kind", ["background", "zero", "rest", "tiny", "large", "waves"])
@pytest.mark.parametrize("limiter", [3, 4])
def test_states_that_choose_either_path(kind, limiter):
    rng = np.random.default_rng(7)
    for rho0, K0 in ((1.0, 4.0), (1.2, 1.4e5), (3.0e-9, 2.0e7)):
        c = np.sqrt(K0 / rho0)
        for nu in (0.0, 0.3, 0.95, 1.2):
            q = _field(kind, 70, 50, rng)
            if kind not in ("background", "rest"):
                q[1:] /= np.sqrt(K0 * rho0)
            _check(q, 0.02, 0.02, nu * 0.02 / c, limiter, 2, 2, rho0, K0, (32, 32, 1, 256))


@pytest.mark.parametrize("limiter", [1, 2, 3, 4])
def test_scaling_by_powers_of_two_crosses_into_the_fp64_phases(limiter):
    # the step is homogeneous and a power of two scales exactly; 2^-600 and 2^600 are outside the
    # exponents that fixed point takes
    q = _field("noise", 45, 37, np.random.default_rng(5))
    base, _ = _step(q, 0.02, 0.02, 0.004, limiter, 2, 2, 1.0, 4.0, (32, 32, 1, 256))
    for k in (-600, 600):
        out, status = _step(np.ldexp(q, k), 0.02, 0.02, 0.004, limiter, 2, 2, 1.0, 4.0, (32, 32, 1, 256))
        assert status == claw.CLAW_OK
        assert np.abs(np.ldexp(out, -k) - base).max() <= TOL * 2.0 * np.abs(q).max()


def test_non_finite_states_are_reported():
    for bad in (np.nan, np.inf, -np.inf):
        q = _field("waves", 40, 40, None)
        q[1, 20, 21] = bad
        got, status = _step(q, 0.02, 0.02, 0.004, 4, 2, 2, 1.0, 4.0, (32, 16, 1, 256))
        assert status == claw.CLAW_ENAN and not np.isfinite(got[:, 15:22, 16:23]).all()
        assert np.isfinite(got[:, 30:, 30:]).all()


def test_error_against_extended_precision_is_no_larger_than_one_rounding_of_the_state():
    # the step in long double (64-bit mantissa or more) of the same doubles: the largest error of each
    # component stays below 1.5 roundings (2^-53) of its largest value, the last of them the result's own
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision on this machine")
    rng = np.random.default_rng(3)
    for kind in ("waves", "noise"):
        q = _field(kind, 64, 48, rng)
        got, status = _step(q, 0.02, 0.02, 0.009, 4, 2, 2, 1.0, 4.0, (32, 16, 1, 256))
        want = _long_step(q.astype(np.longdouble), np.longdouble(0.009) / np.longdouble(0.02))
        err = np.abs(got - want).max(axis=(1, 2)).astype(float)
        assert status == claw.CLAW_OK
        assert np.all(err <= 1.5 * 2.0 ** -53 * np.abs(q).max(axis=(1, 2)).max()), err


def _long_step(q, lam):
    """MC, second order, full transverse corrections, rho = 1, K = 4, dx = dy, in q's own precision"""
    Z, c = q.dtype.type(2), q.dtype.type(2)

    def lim(a, b):
        m, t = np.abs(a), np.where(a < 0, -b, b)
        w = np.where((m > 0) & (t > 0), np.minimum((m + t) / 2, 2 * np.minimum(m, t)), 0)
        return np.where(a < 0, -w, w)

    def sweep(p, u):
        dp, du = np.diff(p, axis=1), np.diff(u, axis=1)
        a1, a2 = (du - dp / Z) / 2, (du + dp / Z) / 2
        m1, m2 = lim(a1[:, 1:-1], a1[:, 2:]), lim(a2[:, 1:-1], a2[:, :-2])
        a1, a2 = a1[:, 1:-1], a2[:, 1:-1]
        k = c * (1 - lam * c) / 2
        fp, fu = k * Z * (m2 - m1), k * (m1 + m2)
        lp, lu, rp, ru = c * Z * a1, -c * a1, c * Z * a2, c * a2
        up = rp[:, :-1] - fp[:, :-1] + lp[:, 1:] + fp[:, 1:]
        uu = ru[:, :-1] - fu[:, :-1] + lu[:, 1:] + fu[:, 1:]
        return up, uu, rp[:, :-1] - 2 * fp[:, :-1] + lp[:, 1:] + 2 * fp[:, 1:]

    def trans(d):
        w = -lam / (4 * Z)
        return w * 4 * (d[:-1] - d[1:]), w * c * (d[:-1] + d[1:])

    xp, xu, D = sweep(q[0], q[1])
    yp, yv, E = (t.T for t in sweep(q[0].T, q[2].T))
    gp, gv = trans(D[1:-1])
    fp, fu = (t.T for t in trans(E[:, 1:-1].T))
    i = slice(2, -2)
    return np.stack([q[0, i, i] - lam * (xp[i] + yp[:, i] + np.diff(fp, axis=1) + np.diff(gp, axis=0)),
                     q[1, i, i] - lam * (xu[i] + np.diff(fu, axis=1)),
                     q[2, i, i] - lam * (yv[:, i] + np.diff(gv, axis=0))])


@pytest.mark.parametrize("medium", [False, True])
@pytest.mark.parametrize("limiter", [0, 1, 2, 3, 4])
def test_cells_out_of_a_disturbance_s_reach_do_not_change(limiter, medium):
    # one disturbed cell in a state of rest on a large pressure: q_new is q bit for bit outside the
    # stencil (two cells in each direction), and zero velocities stay exactly zero there
    n = 40
    run = inputs.Run(0.0, 0.0, 1.0, 1.0, limiter=limiter)
    run.levels = [inputs.Level(n, n, 1.0 / n, 1.0 / n, [(0, 0, n, n)])]
    pool = np.zeros(run.levels[0].qsize)
    q = inputs.box_view(pool, 0, n, n, 3)
    q[0] = 1.0
    q[0, 22, 17] = 1.25
    q[1, 22, 17] = 0.125
    kw = dict(rho0=1.0, K0=4.0)
    args = []
    if medium:
        args = [[[inputs.coef_pool(run.levels[0], f, 1)]] for f in
                (inputs.smooth_field(1, n, n, 0.5, 2.0), inputs.smooth_field(2, n, n, 1.0, 8.0))]
        kw = {}
    H = Hierarchy([run], [[pool]], *args, **kw)
    H.init_dt()
    claw.claw_level_step(H.ctx, 0, H.q[0][0], H.q[0][1], H.aux[0], H.dt, H.smax)
    new = H.interior(0, 0, 0, pool=H.q[0][1])
    old = q[:, 2:-2, 2:-2]
    far = np.ones((n, n), dtype=bool)
    far[18:23, 13:18] = False
    assert np.array_equal(new[:, far], old[:, far]) and not np.array_equal(new, old)
    assert H.sync_status() == claw.CLAW_OK
