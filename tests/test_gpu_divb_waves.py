"""Face divergence of FP32 grids whose blocks take several groups of 256 cells (more than
8 per SM): from the second on, cells that an FP32 bound puts below the largest value so
far are skipped.  The largest value stands early, late, among near ties, in a field
that cancels to its rounding errors, and at cell widths far outside the usual.

The value is FP64 arithmetic of the FP32 faces: six roundings of the terms, as in the
reference."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

DIMS = [(96, 96, 96), (97, 91, 101), (160, 33, 77)]


def _div(st):
    t = [(np.roll(c, -1, ax) - c) / h for c, ax, h in ((st.bx, 2, st.dx), (st.by, 1, st.dy), (st.bz, 0, st.dz))]
    return np.abs(t[0] + t[1] + t[2]), max(np.abs(v).max() for v in t)


def _check(g, st):
    d, m = g.div_b()
    ref, terms = _div(st)
    assert m == max(np.abs(c).max() for c in (st.bx, st.by, st.bz))
    assert abs(d - ref.max()) <= 8 * 2.0 ** -52 * terms, (d, ref.max())


def _state(dims, kind, rng, dx=1 / 64):
    from paper_1808_10633_gb300 import inputs

    nx, ny, nz = dims
    st = inputs.uniform(nx, ny, nz, dx=dx, dy=1.25 * dx, dz=0.75 * dx)
    b = rng.standard_normal((3, nz, ny, nx))
    if kind == "early":
        b *= np.linspace(10, 1, nz)[:, None, None]
    elif kind == "late":
        b *= np.linspace(1, 10, nz)[:, None, None]
    elif kind == "ties":                       # a saw of one height, apart by the last FP32 bits
        b = 1e-6 * b
        b[0] += np.arange(nx) % 2
    else:                                      # div b = 0 up to the rounding of the faces
        A = [sum(np.roll(a, s, ax) for ax in range(3) for s in range(4)) for a in b]
        b = np.stack(inputs.curl_faces(*A, st.dx, st.dy, st.dz)) + 3.0
    return st, b


def _set(st, b):
    st.bx, st.by, st.bz = b.astype(np.float32).astype(np.float64)
    return st


@pytest.mark.parametrize("dims", DIMS)
@pytest.mark.parametrize("kind", ["early", "late", "ties", "cancel"])
def test_periodic_grids(dims, kind):
    from paper_1808_10633_gb300 import wombat as wb

    st = _set(*_state(dims, kind, np.random.default_rng(dims[0])))
    with wb.Grid.from_state(st, precision="fp32") as g:
        _check(g, st)


@pytest.mark.parametrize("kind", ["early", "late", "cancel"])
def test_linked_bricks(kind):
    from paper_1808_10633_gb300 import wombat as wb

    st = _set(*_state((97, 91, 101), kind, np.random.default_rng(2)))
    with wb.Grid.from_bricks(st, ([0, 40, 97], [0, 3, 91], [0, 30, 64, 101]), precision="fp32") as g:
        _check(g, st)


@pytest.mark.parametrize("dx,scale", [(1e46, 1e35), (1e41, 1e30), (1e33, 1e25), (1e-30, 1e-20), (1e-38, 1e30)])
def test_cell_widths_outside_the_fp32_range(dx, scale):
    from paper_1808_10633_gb300 import wombat as wb

    st, b = _state((96, 96, 96), "late", np.random.default_rng(4), dx)
    _set(st, b * scale)
    with wb.Grid.from_state(st, precision="fp32") as g:
        _check(g, st)
