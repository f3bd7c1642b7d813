"""The kernels' own reciprocals and roots (slab_internal.cuh) against exact values, over all exponents, and a factor whose
pivots lie beyond the range of the hardware's approximation."""
import ctypes
import os
import subprocess

import numpy as np
import pytest
import torch

from paper_2211_07572_gb300 import build, inputs

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "slab_internal.cuh"
template <typename T, typename F> __global__ void apply(const T* x, T* y, int n, F f) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = f(x[i]);
}
#define ENTRY(name, T, expr)                                                                        \
    extern "C" int name(const T* x, T* y, int n) {                                                  \
        apply<<<(n + 255) / 256, 256>>>(x, y, n, [] __device__(T v) -> T { return expr; });         \
        return (int)cudaDeviceSynchronize();                                                        \
    }
ENTRY(rcp64, double, reciprocal_full(v))
ENTRY(rsqrt64, double, rsqrt_newton(v))
ENTRY(rcp32, float, reciprocal(v))
ENTRY(rsqrt32, float, rsqrt_newton(v))
ENTRY(rsqrt_tile32, float, rsqrt_tile(v))
__global__ void quotients(const float* a, const float* p, float* y, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = pivot_quotient(a[i], p[i], __float_as_uint(p[i]) & 0x7fffffffu);
}
extern "C" int quotient(const float* a, const float* p, float* y, int n) {
    quotients<<<(n + 255) / 256, 256>>>(a, p, y, n);
    return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("reciprocals")
    src, so = str(d / "r.cu"), str(d / "r.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build.NVCC] + build.CFLAGS + ["--extended-lambda", "-shared", "-o", so, src], check=True)
    return ctypes.CDLL(so)


def _mantissas(dtype, exponents):
    """64 random mantissas, 1 and the one below 2 at every exponent, positive."""
    rng = np.random.default_rng(5)
    m = np.concatenate([[1.0, np.nextafter(dtype(2.0), dtype(0.0))], rng.uniform(1.0, 2.0, 64)]).astype(dtype)
    return np.ldexp(m[None, :], np.asarray(exponents)[:, None]).astype(dtype).reshape(-1)


def _run(fn, *x):
    t = [torch.from_numpy(v).cuda() for v in x]
    y = torch.empty_like(t[0])
    assert fn(*[ctypes.c_void_p(v.data_ptr()) for v in t + [y]], len(x[0])) == 0
    return y.cpu().numpy()


def _units(got, want):
    """Error in units in the last place of the exact value (`want`, long double)."""
    unit = np.spacing(np.abs(want.astype(got.dtype))).astype(np.longdouble)
    return float((np.abs(got.astype(np.longdouble) - want) / unit).max())


# Error bounds: the last Newton step of a reciprocal is one rounding of r + r (1 - x r), whose second term is below 2^-19
# (2^-39) of r and exact to its own rounding: half a unit, and less than one with what is left.  The roots round a r
# (half a unit of the residual, half of that in r) before the last rounding: one unit; beyond the cut-offs stands the library's
# function.  The product form r (1.5 - a r^2 / 2) rounds three times: two.
def test_fp64_reciprocal(lib):
    x = _mantissas(np.float64, range(-1022, 1024))          # through both cut-offs of the Newton form
    x = np.concatenate([x, -x])
    with np.errstate(over="ignore"):
        want = np.longdouble(1) / x.astype(np.longdouble)
    fine = np.abs(want) <= np.longdouble(np.finfo(np.float64).max)
    got = _run(lib.rcp64, x)
    assert _units(got[fine], want[fine]) <= 1.0
    cut = np.concatenate([np.ldexp([1.0, np.nextafter(1.0, 0.0)], e) for e in (-1007, 993)])
    assert _units(_run(lib.rcp64, cut), np.longdouble(1) / cut.astype(np.longdouble)) <= 1.0
    sub = np.array([5e-324, 1e-310, 2.2250738585072009e-308, -1e-309])
    with np.errstate(over="ignore"):
        np.testing.assert_array_equal(_run(lib.rcp64, sub), 1.0 / sub)


def test_fp64_root(lib):
    x = _mantissas(np.float64, range(-1022, 1024))
    want = np.longdouble(1) / np.sqrt(x.astype(np.longdouble))
    got = _run(lib.rsqrt64, x)
    newton = (x >= 2.0 ** -1007) & (x < 2.0 ** 993)
    assert _units(got[newton], want[newton]) <= 1.0
    assert _units(got[~newton], want[~newton]) <= 2.0
    sub = np.array([5e-324, 1e-310, 2.2250738585072009e-308])
    assert _units(_run(lib.rsqrt64, sub), np.longdouble(1) / np.sqrt(sub.astype(np.longdouble))) <= 2.0


def test_fp32(lib):
    x = _mantissas(np.float32, range(-126, 126))            # the reciprocal's range
    x = np.concatenate([x, -x])
    assert _units(_run(lib.rcp32, x), np.longdouble(1) / x.astype(np.longdouble)) <= 1.0
    x = _mantissas(np.float32, range(-125, 128))
    want = np.longdouble(1) / np.sqrt(x.astype(np.longdouble))
    assert _units(_run(lib.rsqrt32, x), want) <= 1.0
    assert _units(_run(lib.rsqrt_tile32, x), want) <= 2.0


def test_fp32_pivot_quotient(lib):
    """|a| <= |p| at every exponent of p, subnormal and above 2^126 too; quotients that are normal numbers."""
    p = np.concatenate([_mantissas(np.float32, range(-126, 128)), np.ldexp(np.float32([1, 3, 5, 1000003]), -149)])
    rng = np.random.default_rng(6)
    a = (p * rng.uniform(-1.0, 1.0, p.size)).astype(np.float32)
    a[::7] = p[::7]
    want = a.astype(np.longdouble) / p.astype(np.longdouble)
    fine = np.abs(want) >= np.finfo(np.float32).tiny
    got = _run(lib.quotient, a, p)
    assert _units(got[fine], want[fine]) <= 2.0             # the reciprocal's unit, and the product's half


@pytest.mark.parametrize("e", [0, 100, 124, 125])
def test_factor_with_large_pivots(e):
    """A convection operator scaled by 2^e: its solution with the load scaled alike is the same, and at e = 125 the pivots
    of the FP32 interface elimination lie above 2^126."""
    from paper_2211_07572_gb300.solver import SlabSolver
    n, b = 128, 8
    x = np.linspace(0.0, 1.0, n + 1)
    kappa = 1.0 + 0.1 * np.outer(np.cos(5 * x), np.sin(6 * x))
    beta = 20.0 * np.stack([np.broadcast_to(np.cos(3 * x), (n + 1, n + 1)), np.broadcast_to(np.sin(2 * x)[:, None], (n + 1, n + 1))])
    f = torch.from_numpy(inputs.normal_rhs(2, n, 2, 3)).cuda()
    s = SlabSolver(2, n, b, inputs.CONVECTION, kappa=np.ldexp(kappa, e), beta=np.ldexp(beta, e), precision="fp32")
    _, rel, _ = s.solve(f * 2.0 ** e)
    s.close()
    assert rel.max() <= 1e-10
