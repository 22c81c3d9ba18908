"""Rounding of the Jiang-Shu and WENO-Z arithmetic of the sweeps (csrc/wb_sweep_js.cuh),
FP32 as the library compiles it and FP64, on stencils given to the functions directly.

u is half a unit in the last place.  e_k = (eps + IS_k) / 16 is a sum of two squares
and eps: the inner difference, its square's term and the sum round three times, the
products of the second square twice, so 4 u of the value holds for any stencil.

A WENO-Z stencil (a, b, b, a) has IS_0 = IS_2 and takes the linear weights, at any size
of IS_1: six roundings of each weight's ratio, two of p and q (each at most four times
the largest difference m), on both sides, over six: 16 u m."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = r'''
#include "wb_sweep_js.cuh"
using namespace wb;
__global__ void kf(const float* x, float* e, float* z, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    constexpr float eps16 = 4.0f * 1e-6f / 16.0f;
    float v[8];
    for (int k = 0; k < 8; k++) v[k] = x[k * n + i];
    float2 e0, e1, e2;
    smoothness<float2>(make_float2(v[0], v[4]), make_float2(v[1], v[5]), make_float2(v[2], v[6]),
                       make_float2(v[3], v[7]), eps16, e0, e1, e2);
    e[i] = e0.x; e[n + i] = e1.x; e[2 * n + i] = e2.x;
    e[3 * n + i] = e0.y; e[4 * n + i] = e1.y; e[5 * n + i] = e2.y;
    const float m[4] = {v[3], v[2], v[1], v[0]}, p[4] = {v[4], v[5], v[6], v[7]};
    z[i] = JsWeights<false>().corr_s(p, m);
    z[n + i] = JsWeights<true>().corr_s(p, m);
}
__global__ void kd(const double* x, double* e, double* z, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    constexpr double eps16 = 4.0 * 1e-6 / 16.0;
    double v[8];
    for (int k = 0; k < 8; k++) v[k] = x[k * n + i];
    for (int s = 0; s < 2; s++)
        smoothness<double>(v[4 * s], v[4 * s + 1], v[4 * s + 2], v[4 * s + 3], eps16, e[3 * s * n + i],
                           e[(3 * s + 1) * n + i], e[(3 * s + 2) * n + i]);
    const double m[4] = {v[3], v[2], v[1], v[0]}, p[4] = {v[4], v[5], v[6], v[7]};
    z[i] = weno_corr<false>(p, m);
    z[n + i] = weno_corr<true>(p, m);
}
template <class T, class K> int go(K k, const T* x, T* o, int n) {
    T* d = nullptr;
    if (cudaMalloc(&d, sizeof(T) * 16 * n) != cudaSuccess) return 1;
    cudaMemcpy(d, x, sizeof(T) * 8 * n, cudaMemcpyHostToDevice);
    k<<<(n + 127) / 128, 128>>>(d, d + 8 * n, d + 14 * n, n);
    const cudaError_t e = cudaMemcpy(o, d + 8 * n, sizeof(T) * 8 * n, cudaMemcpyDeviceToHost);
    cudaFree(d);
    return e == cudaSuccess ? 0 : 2;
}
extern "C" int run_f(const float* x, float* o, int n) { return go<float>(kf, x, o, n); }
extern "C" int run_d(const double* x, double* o, int n) { return go<double>(kd, x, o, n); }
'''


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    from paper_1808_10633_gb300 import build

    d = tmp_path_factory.mktemp("weno")
    src, so = d / "w.cu", d / "w.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.flags(), *build.EXTRA["wb_sweep_f32.cu"], "-I", build.CSRC, "-shared",
                    "-o", str(so), str(src)], check=True)
    return ctypes.CDLL(str(so))


def _run(lib, x, weights="z"):
    """(e of both stencils (6, n), correction (n,)) of x (8, n): two stencils (minus,
    plus side) of four differences, as the kernels take them (doubled)."""
    x = np.ascontiguousarray(x)
    n = x.shape[1]
    out = np.empty((8, n), dtype=x.dtype)
    f = lib.run_f if x.dtype == np.float32 else lib.run_d
    assert f(ctypes.c_void_p(x.ctypes.data), ctypes.c_void_p(out.ctypes.data), ctypes.c_int(n)) == 0
    return out[:6], out[6 + (weights == "z")]


def _indicators(a, b, c, d):
    """eps + IS_0..2 of halved differences, in extended precision."""
    a, b, c, d = (v.astype(np.longdouble) / 2 for v in (a, b, c, d))
    eps = np.longdouble(1e-6)
    return (eps + 13 * (a - b) ** 2 + 3 * (a - 3 * b) ** 2, eps + 13 * (b - c) ** 2 + 3 * (b + c) ** 2,
            eps + 13 * (c - d) ** 2 + 3 * (3 * c - d) ** 2)


def _phi(x, weights):
    """phi_N of halved differences with Jiang-Shu or WENO-Z weights, in extended precision."""
    e = _indicators(*x)
    a = [1 / v ** 2 if weights == "js" else 1 + np.abs(e[0] - e[2]) / v for v in e]
    w = a[0] + 6 * a[1] + 3 * a[2]
    a, b, c, d, w0, w2 = *(v.astype(np.longdouble) / 2 for v in x), a[0] / w, 3 * a[2] / w
    return w0 * (a - 2 * b + c) / 3 + (w2 - 0.5) * (b - 2 * c + d) / 6


U = {np.float32: 2.0 ** -24, np.float64: 2.0 ** -53}
N = 20_000


def _stencils(kind, rng):
    if kind == "random":
        return rng.standard_normal((8, N))
    if kind == "scales":
        return rng.standard_normal((8, N)) * 10.0 ** rng.uniform(-6, 4, (8, N))
    if kind == "least":                       # the directions in which the forms are smallest
        x = rng.standard_normal((8, N)) * 10.0 ** rng.uniform(-3, 3, N)
        for s in (0, 4):
            x[s] = x[s + 1] * (1.375 + rng.uniform(-0.05, 0.05, N))
            x[s + 3] = x[s + 2] * (1.375 + rng.uniform(-0.05, 0.05, N))
        return x
    k, ph = rng.uniform(0.02, 2.0, N), rng.uniform(0, 2 * np.pi, N)
    v = np.sin(k * np.arange(9)[:, None] + ph) * 10.0 ** rng.uniform(-3, 3, N)
    return np.diff(v, axis=0)


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("kind", ["random", "scales", "least", "waves"])
def test_indicators_keep_their_bits(lib, dtype, kind):
    x = _stencils(kind, np.random.default_rng(4)).astype(dtype)
    e, _ = _run(lib, x)
    for s in (0, 1):
        for k, ref in enumerate(_indicators(*x[4 * s:4 * s + 4])):
            rel = np.abs(e[3 * s + k].astype(np.longdouble) / (ref / 4) - 1)
            # the rounded constant 4 eps / 16 is one more u where eps rules
            assert float(rel.max()) <= 5 * U[dtype], (s, k, float(rel.max()) / U[dtype])


@pytest.mark.parametrize("dtype", [np.float32, np.float64])
@pytest.mark.parametrize("size", [1.0, 100.0, 1e4])
def test_weno_z_on_symmetric_stencils(lib, dtype, size):
    rng = np.random.default_rng(5)
    a = size * rng.standard_normal((2, N))
    b = a * np.exp(rng.uniform(-9, 0, (2, N))) * rng.choice([-1, 1], (2, N))
    x = np.stack([a[0], b[0], b[0], a[0], a[1], b[1], b[1], a[1]]).astype(dtype)
    _, z = _run(lib, x)
    err = np.abs(z.astype(np.longdouble) - (_phi(x[:4], "z") - _phi(x[4:], "z")))
    m = np.abs(x).max(axis=0)
    assert float((err / m).max()) <= 16 * U[dtype], float((err / m).max()) / U[dtype]


@pytest.mark.parametrize("weights", ["js", "z"])
@pytest.mark.parametrize("dtype", [np.float32, np.float64])
def test_corrections_at_a_jump(lib, dtype, weights):
    """A jump J seen by both sides where neither takes it into its stencil: each side
    is J / 12 with all but saturated weights and the correction their small difference.  Four
    roundings a side (the numerator's two, the quotient's two) at u / sqrt(3) each are
    1.25 u J rms at most, two sides, over 24 for the halved differences."""
    rng = np.random.default_rng(6)
    j = 10.0 ** rng.uniform(1.5, 3, N)
    x = np.zeros((8, N))
    x[1] = -j * (1 + 1e-3 * rng.standard_normal(N))     # minus side: b
    x[7] = j                                            # plus side: d
    x = x.astype(dtype)
    got = _run(lib, x, weights)[1]
    want = _phi(x[:4], weights) - _phi(x[4:], weights)
    err = (got.astype(np.longdouble) - want) / np.abs(x[7])
    rms = float(np.sqrt((err ** 2).mean()))
    assert rms <= 2 ** 0.5 * 1.25 / 24 * U[dtype], rms / U[dtype]


@pytest.mark.parametrize("precision,dtype", [("fp32", np.float32), ("fp64", np.float64)])
@pytest.mark.parametrize("dims", [(2, 3, 2), (2, 3, 1)])
def test_central_flux_of_uniform_states(precision, dtype, dims):
    """The mass flux of a uniform state is its momentum: the central combination
    (7 (F + F) - (F + F)) / 12 is off by the constant's half u, and no bias else."""
    from paper_1808_10633_gb300 import inputs
    from paper_1808_10633_gb300 import wombat as wb

    rng = np.random.default_rng(7)
    sts, m = [], []
    for _ in range(400):
        st = inputs.uniform(*dims)
        mom = np.exp2(rng.uniform(-2, 0, 3)).astype(dtype).astype(np.float64)
        st.U[0] = 1.0
        st.U[1:4] = mom[:, None, None, None]
        st.U[7] = 10.0
        sts.append(st)
        m.append(mom)
    n, m = dims[0] * dims[1] * dims[2], np.array(m)
    with wb.Grid.from_patches(sts, precision=precision) as g:
        F = [g.face_fluxes(a).reshape(400, 7, n)[:, 0, 0] for a in range(3)]      # patch by patch
    err = np.concatenate([(F[a] - m[:, a]) / m[:, a] for a in range(3)]) / U[dtype]
    assert np.abs(err).max() <= 2.5 and abs(err.mean()) <= 0.6, (err.min(), err.max(), err.mean())
