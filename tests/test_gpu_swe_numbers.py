"""The shallow-water step's building blocks by element, against extended precision: compiled into a
small library of their own from the kernel's header."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1808_02638_gb300 import build

pytestmark = pytest.mark.gpu

LD = np.longdouble
SOURCE = r"""
#include "claw_step_swe.cuh"
__global__ void numbers_kernel(int n, const double* x, double* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    out[i] = claw::swe::recip(x[i]);
    out[n + i] = claw::swe::half(x[i]);
    out[2 * n + i] = claw::swe::twice(x[i]);
}
extern "C" int numbers(int n, const double* x, double* out)
{
    numbers_kernel<<<(n + 255) / 256, 256>>>(n, x, out);
    return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("swe_numbers")
    src, so = str(d / "swe_numbers.cu"), str(d / "swe_numbers.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I" + build.CSRC, "-shared", "-o", so, src], check=True)
    return ctypes.CDLL(os.path.abspath(so))


def _call(fn, *arrays, outs=1):
    import torch
    t = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrays]
    out = torch.empty(outs * t[0].numel(), dtype=torch.float64, device="cuda")
    assert fn(t[0].numel(), *(ctypes.c_void_p(a.data_ptr()) for a in t), ctypes.c_void_p(out.data_ptr())) == 0
    return out.cpu().numpy().reshape(outs, -1)


@pytest.mark.skipif(np.finfo(LD).nmant < 63, reason="no extended precision")
def test_reciprocals_over_exponents_and_mantissa_patterns(lib):
    # the last rounding, 2^-53 of the result at most, and the step's remainder, below 2^-57 of it (2^-56 here:
    # its rounding); operands just below a step of the upper word are the approximation's worst
    rng = np.random.default_rng(0)
    lo = np.array([0, 1, 0x7fffffff, 0x80000000, 0xfffffffe, 0xffffffff], dtype=np.uint64)
    hi = rng.integers(0, 1 << 20, 4000, dtype=np.uint64)
    hi[:6] = [0, 1, (1 << 20) - 1, (1 << 20) - 2, 1 << 19, (1 << 19) - 1]
    m = np.concatenate([((hi[:, None] << np.uint64(32)) | lo).ravel(),
                        rng.integers(0, 1 << 52, 200_000, dtype=np.uint64)])
    e = rng.integers(1, 2045, m.size).astype(np.uint64)
    e[:2 * hi.size] = 1023
    x = ((e << np.uint64(52)) | m).view(np.float64)
    got = _call(lib.numbers, x, outs=3)[0]
    rel = np.abs(got.astype(LD) * x.astype(LD) - 1)
    assert np.all(rel <= LD(2.0 ** -53 + 2.0 ** -56)), float(rel.max())
    assert np.array_equal(_call(lib.numbers, -x, outs=3)[0], -got)


def test_halves_and_doubles_and_what_is_not_finite(lib):
    rng = np.random.default_rng(1)
    x = np.ldexp(rng.uniform(1.0, 2.0, 10_000), rng.integers(-1020, 1022, 10_000)) * rng.choice([-1.0, 1.0], 10_000)
    x = np.concatenate([x, [0.0, -0.0, 2.0 ** -1021, 2.0 ** 1022, -(2.0 ** 1022)]])
    r, h, d = _call(lib.numbers, x, outs=3)
    assert np.array_equal(h, 0.5 * x) and np.array_equal(d, 2.0 * x)
    assert np.array_equal(np.signbit(h), np.signbit(x)) and np.array_equal(np.signbit(d), np.signbit(x))
    r, h, d = _call(lib.numbers, np.array([np.inf, -np.inf, np.nan, -np.nan]), outs=3)
    assert np.array_equal(r[:2], [0.0, 0.0]) and np.isnan(r[2:]).all()
    for y in (h, d):
        assert np.array_equal(y[:2], [np.inf, -np.inf]) and np.isnan(y[2:]).all()
    assert not np.isfinite(_call(lib.numbers, np.array([0.0]), outs=3)[0])


@pytest.mark.parametrize("component", [0, 1, 2])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_states_that_are_not_finite_are_reported(bad, component):
    from paper_1808_02638_gb300 import claw, inputs
    from paper_1808_02638_gb300.solver import Hierarchy
    n = 40
    run = inputs.Run(0.0, 0.0, 1.0, 1.0)
    run.levels = [inputs.Level(n, n, 1.0 / n, 1.0 / n, [(0, 0, n, n)])]
    pool = np.zeros(run.levels[0].qsize)
    q = inputs.box_view(pool, 0, n, n, 3)
    q[0], q[1], q[2] = 1.0, 0.2, -0.1
    q[component, 20, 21] = bad
    H = Hierarchy([run], [[pool]], system="shallow_water", grav=1.0)
    H.dt.fill_(0.2 / n)
    claw.claw_level_step(H.ctx, 0, H.q[0][0], H.q[0][1], None, H.dt, H.smax)
    new = H.interior(0, 0, 0, pool=H.q[0][1])
    assert H.sync_status() == claw.CLAW_ENAN
    assert not np.isfinite(new[:, 18, 19]).all() and np.isfinite(new[:, :10]).all() and np.isfinite(new[:, 30:]).all()
    H.close()
