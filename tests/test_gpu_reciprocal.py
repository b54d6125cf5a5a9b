"""The reciprocals and inverse roots of the kernels against exact values over their argument range, at the range's
ends, and what a caller sees of them where a density is zero.

Bounds.  rcp_s: the refined value is rounded once, what the series leaves is of order 2^-60: 1 ulp.  rsqrt_s: half an
ulp from the last rounding, half at most from that of x y: 1 ulp and the same remainder, 1.1.  FP32: those that the
PTX documentation states for the instructions, 1 ulp and 2^-22.9."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_1810_07802_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "dugks_strip.cuh"
template <typename F, typename T> __global__ void map(F f, const T *x, T *y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = f(x[i]);
}
struct Rcp64 { __device__ double operator()(double v) const { return dugks::rcp_s(v); } };
struct Root64 { __device__ double operator()(double v) const { return dugks::rsqrt_s(v); } };
struct Rcp32 { __device__ float operator()(float v) const { return dugks::rcp_r(v); } };
struct Root32 { __device__ float operator()(float v) const { return dugks::rsqrt_r(v); } };
struct CudaRcp32 { __device__ float operator()(float v) const { return __fdividef(1.0f, v); } };
struct CudaRoot32 { __device__ float operator()(float v) const { return rsqrtf(v); } };
template <typename F, typename T> int run(F f, const T *x, T *y, int n) {
    map<<<(n + 255) / 256, 256>>>(f, x, y, n);
    return (int)cudaDeviceSynchronize();
}
extern "C" int rcp64(const double *x, double *y, int n) { return run(Rcp64(), x, y, n); }
extern "C" int root64(const double *x, double *y, int n) { return run(Root64(), x, y, n); }
extern "C" int rcp32(const float *x, float *y, int n) { return run(Rcp32(), x, y, n); }
extern "C" int root32(const float *x, float *y, int n) { return run(Root32(), x, y, n); }
extern "C" int cuda_rcp32(const float *x, float *y, int n) { return run(CudaRcp32(), x, y, n); }
extern "C" int cuda_root32(const float *x, float *y, int n) { return run(CudaRoot32(), x, y, n); }
"""


@pytest.fixture(scope="module")
def call(tmp_path_factory):
    import torch

    from paper_1810_07802_gb300 import build

    d = tmp_path_factory.mktemp("reciprocal")
    src, so = str(d / "map.cu"), str(d / "map.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.nvcc(), "-O3", "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", build.INCLUDE, "-I",
                    build.CSRC, "-o", so, src] + build.ARCH, check=True)
    lib = ctypes.CDLL(so)

    def go(name, x):
        a = torch.from_numpy(x).cuda()
        b = torch.empty_like(a)
        torch.cuda.synchronize()
        assert getattr(lib, name)(ctypes.c_void_p(a.data_ptr()), ctypes.c_void_p(b.data_ptr()), x.size) == 0
        return b.cpu().numpy()

    return go


def arguments(lo, hi, dtype, n=400000):
    """n mantissas, exponents lo .. hi - 1, and every power of two of the range with its neighbours."""
    r = np.random.default_rng(7)
    one = np.ldexp(1.0, np.arange(lo + 1, hi)).astype(dtype)
    x = np.ldexp(1.0 + r.random(n), r.integers(lo, hi, n)).astype(dtype)
    return np.concatenate([x, one, np.nextafter(one, dtype(0)), np.nextafter(one, dtype(np.inf))])


def ulps(got, exact, dtype):
    """|got - exact| in units in the last place of the exact value."""
    return float(np.max(np.abs(got.astype(exact.dtype) - exact) / np.spacing(np.abs(exact).astype(dtype))))


def test_fp64(call):
    x = arguments(-1021, 1021, np.float64)
    x = np.concatenate([x, -x])
    assert ulps(call("rcp64", x), 1 / x.astype(np.longdouble), np.float64) <= 1.0
    x = arguments(-1021, 1023, np.float64)
    assert ulps(call("root64", x), 1 / np.sqrt(x.astype(np.longdouble)), np.float64) <= 1.1


def test_fp64_at_the_ends_of_the_range(call):
    x = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, 5e-324])
    with np.errstate(divide="ignore", over="ignore"):
        want = 1 / x
    got = call("rcp64", x)
    assert np.array_equal(got, want, equal_nan=True) and np.array_equal(np.signbit(got[:4]), np.signbit(want[:4]))
    x = np.array([0.0, np.inf, np.nan, -1.0])
    assert np.array_equal(call("root64", x), np.array([np.inf, 0.0, np.nan, np.nan]), equal_nan=True)


def test_fp32(call):
    x = arguments(-126, 126, np.float32)
    got = call("rcp32", x)
    assert ulps(got, 1 / x.astype(np.float64), np.float32) <= 1.0
    assert np.array_equal(got, call("cuda_rcp32", x))
    got = call("root32", x)
    exact = 1 / np.sqrt(x.astype(np.float64))
    assert float(np.max(np.abs(got - exact) / exact)) <= 2.0 ** -22.9
    assert np.array_equal(got, call("cuda_root32", x))


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
def test_velocity_where_the_density_is_zero(precision):
    """The density 1 + phi is zero at phi = -1: a non-zero momentum over it reads out as an infinite velocity."""
    import torch

    from paper_1810_07802_gb300 import solver

    nx, ny = 8, 5
    cfg, f = W.random_state(nx, ny, seed=1)
    cfg = dict(cfg, rho_h=2.0, rho_l=1.0, gx=0.0, gy=0.0, gravity_mode=0, precision=precision, phi_ref=0.0)
    with solver.Solver(cfg, **f) as s:
        buf = s.row_buffer(ny)
        buf.zero_()
        buf[0] = -1.0
        buf[9 + 1] = 0.125
        buf[9 + 7] = 0.25
        torch.cuda.synchronize()
        s.set_rows(0, ny, buf)
        m = s.macros()
        umax = s.reduce()[3]
    assert np.all(m["phi"] == -1.0)
    assert np.all(m["ux"] == np.inf) and np.all(m["uy"] == -np.inf) and umax == np.inf
