"""The FP64 reciprocal of the step and adjoint kernels (csrc/lbm_fp64.cuh) and
the reciprocal square root of the eigenvalue iteration (csrc/lbm_eig.cuh) on
the device, against extended-precision quotients and CUDA's own functions."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_0706_0405_gb300 import build, lbm
from paper_0706_0405_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_eig.cuh"
#include "lbm_fp64.cuh"
__global__ void k(const double* x, double* y, int n, int which) {
    const int q = blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    const double a = x[q];
    y[q] = which == 0 ? lbm::fp64_rcp(a) : which == 1 ? __drcp_rn(a) : which == 2 ? lbm::rsqrt_pos(a) : rsqrt(a);
}
extern "C" int run(const double* x, double* y, int n, int which) {
    double *dx = nullptr, *dy = nullptr;
    int bad = cudaMalloc(&dx, 8 * (size_t)n) || cudaMalloc(&dy, 8 * (size_t)n) ||
              cudaMemcpy(dx, x, 8 * (size_t)n, cudaMemcpyHostToDevice);
    if (!bad) {
        k<<<(n + 127) / 128, 128>>>(dx, dy, n, which);
        bad = cudaMemcpy(y, dy, 8 * (size_t)n, cudaMemcpyDeviceToHost);
    }
    cudaFree(dx);
    cudaFree(dy);
    return bad;
}
"""
RCP, CUDA_RCP, RSQRT, CUDA_RSQRT = range(4)


@pytest.fixture(scope="module")
def apply(tmp_path_factory):
    d = tmp_path_factory.mktemp("rcp")
    src, lib = d / "harness.cu", d / "libharness.so"
    src.write_text(SOURCE)
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    flags = [f for f in build.FLAGS if f != "-lineinfo"]
    r = subprocess.run([nvcc, *build.ARCH, *flags, "-shared", "-I", build.CSRC, "-I", build.INCLUDE, str(src), "-o",
                        str(lib)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    fn = ctypes.CDLL(str(lib)).run

    def run(which, x):
        x = np.ascontiguousarray(x, dtype=np.float64)
        y = np.empty_like(x)
        ptr = lambda a: a.ctypes.data_as(ctypes.c_void_p)
        assert fn(ptr(x), ptr(y), ctypes.c_int(x.size), ctypes.c_int(which)) == 0
        return y
    return run


def _significands(n):
    """Random ones, those around every 2^-12 of [1, 2) (where a table of the
    approximation may change entries), and the ends."""
    rng = np.random.default_rng(3)
    edges = (1.0 + np.arange(4096) / 4096.0)[:, None] + np.array([-1, 0, 1]) * 2.0 ** -52
    s = np.concatenate([1.0 + rng.random(n), edges.ravel(), [1.0, np.nextafter(2.0, 0.0)]])
    return s[(s >= 1.0) & (s < 2.0)]


def _ulps(got, want):
    """|got - want| in units of the last place of want (extended precision)."""
    return np.abs(got.astype(np.longdouble) - want) / np.spacing(want.astype(np.float64)).astype(np.longdouble)


def test_reciprocal_within_its_bound_for_every_exponent(apply):
    """0.51 ulp: half an ulp of the last rounding and the 2^-60 that the third
    order step leaves of a seed good to 2^-20 (2^-7 ulp at most).  Both signs,
    all exponents whose reciprocals are normal."""
    s = _significands(4000)
    e = np.random.default_rng(4).integers(-1022, 1022, s.size)
    e[:8] = [-1022, -1021, -1, 0, 1, 1020, 1021, 1021]
    for a in (s, np.ldexp(s, e), -np.ldexp(s, e)):
        want = 1.0 / a.astype(np.longdouble)
        got = apply(RCP, a)
        assert _ulps(got, want).max() <= 0.51
        assert (np.abs(got - apply(CUDA_RCP, a)) <= np.spacing(np.abs(got))).all()


def test_reciprocal_outside_that_range(apply):
    """NaN below the normal numbers and at infinity; among the largest, whose
    reciprocals are subnormal, the approximation is flushed to zero (but for
    those next to 2^1022)."""
    a = np.array([0.0, -0.0, 2.0 ** -1074, 2.0 ** -1030, np.nextafter(2.0 ** -1022, 0.0), np.inf, -np.inf, np.nan])
    assert np.isnan(apply(RCP, a)).all()
    assert not apply(RCP, np.array([1.5 * 2.0 ** 1023, -1.5 * 2.0 ** 1023, np.finfo(float).max])).any()


def _state(nx=40, ny=4):
    import torch
    p = W.uniform(nx, ny, (1.0, 0.3, 0.05, 1.0), dx=0.01, sides=(W.Side("outflow"),) * 2 + (W.Side("periodic"),) * 2)
    with lbm.Lattice(p, "fp64") as lat:
        f = lat.init(*W.initial_fields(p, seed=1, sigma=0.05)).get_f()
    return p, f, torch


@pytest.mark.parametrize("k", [-900, 900])
def test_the_step_is_homogeneous_over_the_range_of_densities(k):
    """The update is of degree one in f: scaled by a power of two that leaves
    its products in range, the levels have the same bits, from the kernel of
    one step and from the one of several."""
    p, f, torch = _state()
    out = []
    for scale in (1.0, 2.0 ** k):
        with lbm.Lattice(p, "fp64") as lat:
            lat.set_f(f * scale).step(1).step(5)
            out.append(lat.get_f() / scale)
            assert lat.health() == 0
    assert torch.equal(out[0], out[1])


@pytest.mark.parametrize("rho", [2.0 ** 1022, 1.9 * 2.0 ** 1022, 0.0, -1.0, 2.0 ** -1030, float("inf"), float("nan")])
@pytest.mark.parametrize("steps", [1, 3])
def test_a_density_without_a_reciprocal_is_non_physical(rho, steps):
    """One node of such a density among ordinary ones (all of it at rest, so
    that the sums are exact)."""
    p, f, torch = _state()
    f[:, 2, 17] = 0.0
    f[0, 2, 17] = rho
    with lbm.Lattice(p, "fp64") as lat:
        lat.set_f(f).step(steps)
        assert lat.health() & lbm.LBM_FLAG_NONPHYSICAL
        with pytest.raises(lbm.LbmError) as ei:
            lat.sync()
        assert ei.value.status == lbm.LBM_E_NONPHYSICAL


def test_reciprocal_square_root_within_its_bound(apply):
    """1.03 ulp: half an ulp of the last rounding, half of the rounding of a y
    in the residual, and at most 2^-58 of a seed good to 2^-20 (residual
    2^-19).  From 2^-960, below which the iteration counts a square as zero,
    to 2^960; CUDA's own function to the sum of both bounds (it is stated to 2
    ulp at most)."""
    s = _significands(4000)
    e = np.random.default_rng(5).integers(-960, 960, s.size)
    e[:6] = [-960, -959, -1, 0, 958, 959]
    for a in (s, 2.0 * s, np.ldexp(s, e)):
        want = 1.0 / np.sqrt(a.astype(np.longdouble))
        got = apply(RSQRT, a)
        assert _ulps(got, want).max() <= 1.03
        assert (np.abs(got - apply(CUDA_RSQRT, a)) <= 3.03 * np.spacing(got)).all()
    special = apply(RSQRT, np.array([np.inf, np.nan, -1.0]))
    assert np.isnan(special[1:]).all() and not special[0] > 0.0
