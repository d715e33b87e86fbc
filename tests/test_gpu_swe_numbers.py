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
__global__ void strengths_kernel(int n, const double* un, const double* c, const double* dh, const double* dn, double* out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    double a1, a2, a3;
    claw::swe::strengths(un[i] - c[i], un[i] + c[i], 0.0, 0.5 / c[i], dh[i], dn[i], 0.0, a1, a2, a3);
    out[i] = a1;
    out[n + i] = a3;
}
extern "C" int strengths(int n, const double* un, const double* c, const double* dh, const double* dn, double* out)
{
    strengths_kernel<<<(n + 255) / 256, 256>>>(n, un, c, dh, dn, out);
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
@pytest.mark.parametrize("wave", [1, 3])
def test_the_strength_of_an_absent_wave_is_as_exact_as_its_speed(lib, wave):
    # The jump is all but one wave of the edge's own Roe state, so that the other's strength is a difference
    # that cancels: its error is that of the speed's rounding (2^-53 for a speed below 2) times dh / 2c, and
    # its own relative roundings.  Formed from the present wave's strength it would be that one's: 2^-53 |dh|.
    rng = np.random.default_rng(wave)
    n = 100_000
    h = rng.uniform(0.5, 1.5, n)
    un, c, dh = rng.uniform(-0.3, 0.3, n), np.sqrt(h), h * rng.uniform(-0.6, 0.6, n)
    dn = (un - c if wave == 1 else un + c) * dh * (1.0 + rng.uniform(-1.0e-9, 1.0e-9, n))
    a1, a3 = _call(lib.strengths, un, c, dh, dn, outs=2)
    U, C, H, N = (x.astype(LD) for x in (un, c, dh, dn))
    want1, want3 = ((U + C) * H - N) / (2 * C), (N - (U - C) * H) / (2 * C)
    got, want = (a3, want3) if wave == 1 else (a1, want1)
    err = np.abs(got - want).astype(float)
    assert np.all(err <= 2.0 ** -53 * (np.abs(dh) / (2.0 * c) + 4.0 * np.abs(want).astype(float)))
    other, wanto = (a1, want1) if wave == 1 else (a3, want3)
    assert np.all(np.abs(other - wanto) <= 6.0 * 2.0 ** -53 * np.abs(wanto))
