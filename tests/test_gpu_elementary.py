"""The device functions under every residual and factor: ln_tab (model.cuh) against the logarithm in
extended precision, to a unit in the last place as CUDA's log(), over the normal numbers, next to 1 and
next to the borders of its table, and log()'s own answers elsewhere; cond_recip (kernels_cond.cuh) and
ldl_recip (kernels_ldl.cuh) against division, to a unit in the last place over the ranges that they state.
A small library of kernels that call them is compiled here."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "kernels.cuh"
#include "kernels_warp.cuh"
#include "vec_kernels.cuh"
#include "kernels_cond.cuh"
#include "kernels_ldl.cuh"
using namespace absorber;
__global__ void ln_kernel(int n, const double* x, double* y, double* z) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    y[i] = ln_tab(x[i]);
    z[i] = log(x[i]);
}
template <class T>
__global__ void recip_kernel(int n, const T* x, T* y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = cond_recip(x[i]);
}
__global__ void ldl_recip_kernel(int n, const double* x, double* y) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) y[i] = ldl_recip(x[i]);
}
extern "C" int run(int what, int n, const void* x, void* y, void* z) {
    static LnEntry t[LN_TAB];
    fill_ln_table(t);
    if (cudaMemcpyToSymbol(g_ln, t, sizeof(t)) != cudaSuccess) return 1;
    const int g = (n + 127) / 128;
    if (what == 0) ln_kernel<<<g, 128>>>(n, (const double*)x, (double*)y, (double*)z);
    if (what == 1) recip_kernel<double><<<g, 128>>>(n, (const double*)x, (double*)y);
    if (what == 2) recip_kernel<float><<<g, 128>>>(n, (const float*)x, (float*)y);
    if (what == 3) ldl_recip_kernel<<<g, 128>>>(n, (const double*)x, (double*)y);
    return cudaDeviceSynchronize() != cudaSuccess;
}
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    from paper_2607_15420_gb300 import build
    d = tmp_path_factory.mktemp("elementary")
    src, so = str(d / "elementary.cu"), str(d / "libelementary.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([build._nvcc(), *build.ARCH, "-O2", "-std=c++17", "--expt-relaxed-constexpr", "-shared",
                    "-Xcompiler", "-fPIC", "-I", build.CSRC, "-I", build.INCLUDE, src, "-o", so], check=True)
    lib = C.CDLL(os.path.abspath(so))
    lib.run.argtypes = [C.c_int, C.c_int, C.c_void_p, C.c_void_p, C.c_void_p]

    def call(what, x):
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        y, z = torch.zeros_like(t), torch.zeros_like(t)
        torch.cuda.synchronize()
        assert lib.run(what, t.numel(), t.data_ptr(), y.data_ptr(), z.data_ptr()) == 0
        return y.cpu().numpy(), z.cpu().numpy()

    return call


def _ulps(y, exact, dtype):
    e = exact.astype(dtype)
    return np.abs(y.astype(np.longdouble) - exact) / np.spacing(np.abs(e)).astype(np.longdouble)


def test_logarithm(run):
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision")
    rng = np.random.default_rng(3)
    eps = 2.0 ** -52
    near = np.concatenate([1.0 + k * np.arange(1, 2000) for k in (eps, -eps / 2)]
                          + [1.0 + s * np.exp(-36.0 * rng.random(100000)) * 0.5 for s in (1.0, -1.0)])
    c = 1.0 + (np.arange(0, 257) / 256.0)
    borders = np.concatenate([np.ldexp(np.nextafter(c, t), e) for t in (0.0, 1.0 + c.max()) for e in (-900, -1, 0, 1, 900)]
                             + [np.ldexp(c, e) for e in (-900, -1, 0, 1, 900)])
    x = np.concatenate([np.exp(rng.uniform(-707.0, 709.0, 200000)), np.exp(rng.uniform(-12.0, 12.0, 200000)),
                        rng.uniform(0.5, 2.0, 200000), near, borders, [2.0 ** -1022, np.finfo(np.float64).max]])
    y, _ = run(0, x)
    exact = np.log(x.astype(np.longdouble))
    one = x == 1.0
    assert np.all(y[one] == 0.0)
    assert np.max(_ulps(y[~one], exact[~one], np.float64)) <= 1.0


def test_logarithm_of_other_numbers(run):
    x = np.array([0.0, -0.0, 5e-324, 1e-310, 2.0 ** -1023, -1.0, -1e-310, np.inf, -np.inf, np.nan])
    y, z = run(0, x)
    np.testing.assert_array_equal(y, z)


@pytest.mark.parametrize("what,dtype,top", [(1, np.float64, 1000), (2, np.float32, 124), (3, np.float64, 1000)])
def test_reciprocal(run, what, dtype, top):
    rng = np.random.default_rng(4)
    e = np.concatenate([rng.integers(-top, top, 300000), np.arange(-top, top)])
    m = np.concatenate([rng.uniform(1.0, 2.0, 300000), np.ones(2 * top)])
    m[:1000] = np.nextafter(dtype(2.0), dtype(0.0))
    m[1000:2000] = np.nextafter(dtype(1.0), dtype(2.0))
    x = (np.ldexp(m, e) * np.where(rng.random(e.size) < 0.5, -1.0, 1.0)).astype(dtype)
    y, _ = run(what, x)
    assert np.max(_ulps(y, 1.0 / x.astype(np.longdouble), dtype)) <= 1.0
