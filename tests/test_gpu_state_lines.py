"""State copies in and out, whose threads follow the 128-byte lines of the host
arrays: patches smaller than a line, of odd sizes and around a block's 256 cells,
host arrays that start anywhere, FP32 and FP64, pinned and pageable.  What was put
in comes out unchanged; the cell-centred field is the rounded mean of its faces."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

DIMS = [(3, 1, 1), (17, 1, 1), (5, 7, 9), (16, 4, 4), (255, 1, 1), (1, 257, 1), (32, 5, 3), (31, 33, 8), (8, 1, 63)]


@pytest.mark.parametrize("pinned", [True, False])
@pytest.mark.parametrize("shift", [0, 1, 13, 31])
@pytest.mark.parametrize("precision,dtype", [("fp32", torch.float32), ("fp32", torch.float64), ("fp64", torch.float64)])
def test_state_comes_back(precision, dtype, shift, pinned):
    from paper_1808_10633_gb300 import wombat as wb

    n = [a * c * d for a, c, d in DIMS]
    N = sum(n)
    rng = np.random.default_rng(4)
    U, b = rng.uniform(1, 2, 8 * N).astype(np.float32), rng.uniform(0.1, 0.2, 3 * N).astype(np.float32)
    for p, m in enumerate(n):
        U[8 * sum(n[:p]) + 7 * m:8 * sum(n[:p + 1])] += 20          # energies: positive pressures

    def place(v):
        t = torch.full((v.size + 64,), -7.0, dtype=dtype, pin_memory=pinned)
        t[shift:shift + v.size] = torch.from_numpy(v).to(dtype)
        return t, t[shift:shift + v.size]

    (_, Ui), (_, bi) = place(U), place(b)
    (Uh, Uo), (bh, bo) = place(0 * U), place(0 * b)
    arg = (lambda t: t) if pinned else (lambda t: t.numpy())
    with wb.Grid(DIMS, 0.1, 0.1, 0.1, np.ones(8 * N) + 20 * (np.arange(8 * N) % 2), np.zeros(3 * N), precision=precision) as g:
        g.set_state(arg(Ui), arg(bi))
        g.get_state(arg(Uo), arg(bo))
        V, c = g.get_state()
    for h, m in ((Uh, 8 * N), (bh, 3 * N)):                          # nothing beside the arrays is touched
        assert (h[:shift] == -7).all() and (h[shift + m:] == -7).all()
    Uo, bo = Uo.numpy(), bo.numpy()
    assert np.array_equal(bo, bi.numpy()) and np.array_equal(c, bi.numpy())
    o = 0
    for (nx, ny, nz), m in zip(DIMS, n):
        want, f = Ui.numpy()[8 * o:8 * (o + m)].reshape(8, nz, ny, nx).copy(), bi.numpy()[3 * o:3 * (o + m)]
        f = f.reshape(3, nz, ny, nx).astype(np.float64)
        for d in range(3):
            want[4 + d] = (0.5 * (f[d] + np.roll(f[d], -1, 2 - d))).astype(want.dtype)
        assert np.array_equal(Uo[8 * o:8 * (o + m)].reshape(want.shape), want)
        assert np.array_equal(V[8 * o:8 * (o + m)].reshape(want.shape).astype(want.dtype), want)
        o += m
