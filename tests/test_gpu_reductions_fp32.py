"""Totals and face divergence of FP32 grids: four values are added in FP32 with
their rounding errors kept, so the sums must match exact ones as FP64 sums do,
for alternating signs that cancel, values over the whole FP32 range, and cell
counts around the four strided values of a thread.

Tolerance of the totals: a thread adds at most 7 groups of four here and the
tree 18 more levels, each rounding at 2^-53 of a partial sum that is at most
the sum of magnitudes: 32 x 2^-53 of that."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _totals(state):
    import torch

    from paper_1808_10633_gb300 import wombat as wb

    d = torch.from_numpy(state).cuda()
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    wb.conserved_totals_noalloc(d.data_ptr(), "fp32", state.shape[1], 1.0, out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()[[0, 1, 2, 3, 7, 4, 5, 6]]


@pytest.mark.parametrize("n", [1, 3, 255, 256, 1023, 1024, 1025, 300_007])
@pytest.mark.parametrize("kind", ["normal", "cancel", "range", "huge"])
def test_fp32_totals_are_exact_sums(n, kind):
    rng = np.random.default_rng(n)
    x = rng.standard_normal((8, n))
    if kind == "cancel":
        x[:, n // 2: 2 * (n // 2)] = -x[:, :n // 2] * (1 + 1e-7)
    elif kind == "range":
        x = x * np.exp2(rng.integers(-140, 100, (8, n)))
    elif kind == "huge":
        x = np.where(rng.uniform(size=(8, n)) < 0.5, 3.2e38, -3.3e38) * rng.uniform(0.9, 1.0, (8, n))
    x = x.astype(np.float32)
    got = _totals(x)
    for f in range(8):
        v = x[f].astype(np.float64)
        assert abs(got[f] - math.fsum(v)) <= 32 * 2.0 ** -53 * math.fsum(np.abs(v)), (f, got[f])


def test_fp32_totals_keep_infinities_and_nan():
    x = np.ones((8, 5000), dtype=np.float32)
    x[0, 1234] = np.inf
    x[1, 77] = -np.inf
    x[2, 10], x[2, 11] = np.inf, -np.inf
    x[3, 4999] = np.nan
    x[4, 3] = 3.4e38
    x[4, 259] = 3.4e38
    got = _totals(x)
    assert got[0] == np.inf and got[1] == -np.inf and np.isnan(got[2]) and np.isnan(got[3])
    assert got[4] == float(np.float32(3.4e38)) * 2 + 4998
    assert np.all(got[5:] == 5000)


@pytest.mark.parametrize("dims", [(33, 7, 5), (64, 64, 64), (1, 1, 1), (129, 2, 1)])
def test_fp32_face_divergence(dims):
    """max |div b| and max |b| of rough face fields against FP64 arithmetic on
    the FP32 values: six roundings of the terms."""
    from paper_1808_10633_gb300 import inputs
    from paper_1808_10633_gb300 import wombat as wb

    nx, ny, nz = dims
    rng = np.random.default_rng(nx)
    st = inputs.uniform(nx, ny, nz)
    b = (rng.standard_normal((3, nz, ny, nx)) * 10.0 ** rng.integers(-3, 2, (3, nz, ny, nx))).astype(np.float32)
    st.bx, st.by, st.bz = (c.astype(np.float64) for c in b)
    with wb.Grid.from_state(st, precision="fp32") as g:
        d, m = g.div_b()
    t = [(np.roll(c, -1, ax) - c) / h for c, ax, h in ((st.bx, 2, st.dx), (st.by, 1, st.dy), (st.bz, 0, st.dz))]
    ref = np.abs(t[0] + t[1] + t[2]).max()
    assert m == np.abs(b).max()
    assert abs(d - ref) <= 8 * 2.0 ** -52 * max(np.abs(v).max() for v in t)
