"""The FP64 reciprocal and (reciprocal) square root of the sweep kernels
(csrc/wb_math.cuh) over the whole range: within one unit in the last place of
the exact value for normal arguments and results, and CUDA's own results for
zero, subnormal, infinite, negative and NaN arguments."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r'''
#include "wb_math.cuh"
__global__ void k(const double* x, double* r, double* q, double* s, double* c, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    r[i] = wb::recip(x[i]);
    q[i] = wb::rsq_root(x[i]);
    s[i] = wb::sq_root(x[i]);
    c[i] = 1.0 / x[i];
    c[n + i] = rsqrt(x[i]);
    c[2 * n + i] = sqrt(x[i]);
}
extern "C" int run(const double* x, double* o, int n) {
    double* d = nullptr;
    if (cudaMalloc(&d, sizeof(double) * 7 * n) != cudaSuccess) return 1;
    cudaMemcpy(d, x, sizeof(double) * n, cudaMemcpyHostToDevice);
    k<<<(n + 255) / 256, 256>>>(d, d + n, d + 2 * n, d + 3 * n, d + 4 * n, n);
    const cudaError_t e = cudaMemcpy(o, d + n, sizeof(double) * 6 * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}
'''


def _run(tmp_path, x):
    from paper_1808_10633_gb300 import build

    src, lib = tmp_path / "m.cu", tmp_path / "m.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.flags(), "-I", build.CSRC, "-shared", "-o", str(lib), str(src)], check=True)
    out = np.empty((6, x.size))
    L = ctypes.CDLL(str(lib))
    assert L.run(ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(out.ctypes.data), ctypes.c_int(x.size)) == 0
    return out


def test_reciprocals_and_roots(tmp_path):
    rng = np.random.default_rng(3)
    n = 1 << 18
    x = np.ldexp(rng.uniform(1.0, 2.0, n), rng.integers(-1022, 1024, n))
    edge = np.ldexp(np.array([1.0, 1.0 + 2.0 ** -52, 2.0 - 2.0 ** -52, 1.5]), np.arange(-1022, 1024)[:, None]).ravel()
    special = np.array([0.0, -0.0, np.inf, -np.inf, np.nan, -1.0, -1e-300, 5e-324, 1e-310, 2.2e-308, 1.79e308])
    x = np.concatenate([x, edge, special])
    with np.errstate(all="ignore"):
        got = _run(tmp_path, x)
        m = slice(0, x.size - special.size)
        big = x[m].astype(np.longdouble)
        for k, ref in enumerate((1 / big, 1 / np.sqrt(big), np.sqrt(big))):
            normal = np.abs(ref) > 2.3e-308
            err = np.abs(got[k][m].astype(np.longdouble) - ref)[normal] / np.spacing(np.abs(ref[normal]).astype(float))
            assert float(err.max()) <= 1.0, (k, float(err.max()))
            sub = ~normal
            assert np.array_equal(got[k][m][sub], got[3 + k][m][sub]), k
            a, b = got[k][-special.size:], got[3 + k][-special.size:]
            both = np.isnan(a) & np.isnan(b)
            near = np.isfinite(b) & (np.abs(a - b) <= np.spacing(np.abs(b)))
            assert np.all(both | (a == b) | near), (k, a, b)
