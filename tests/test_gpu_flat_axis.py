"""Sweeps along an axis of one cell (2-D and 1-D grids) take one thread per
cell: the same state two and eight cells deep along that axis, uniform in it,
goes through the ordinary tiles and must give the same fluxes, and so must a
whole step.  Sizes around the 128 cells of a flat tile.

Tolerance: the fluxes of a uniform axis are the central combination of four
equal values plus a correction of exact zeros, so both paths round a handful of
times: 8 ulp of each component's scale."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = {"fp64": 2.0 ** -52, "fp32": 2.0 ** -23}


def _flat_state(axis, na, nb, seed):
    """A perturbed state one cell deep along `axis`."""
    from paper_1808_10633_gb300 import inputs

    dims = [0, 0, 0]
    dims[axis], dims[(axis + 1) % 3], dims[(axis + 2) % 3] = 1, na, nb
    return inputs.perturbed(*dims, seed=seed, jump=min(na, nb) > 4)


def _deep(st, axis, n):
    from paper_1808_10633_gb300 import inputs

    rep = lambda a: np.repeat(a, n, axis=a.ndim - 1 - axis)
    return inputs.State(rep(st.U), rep(st.bx), rep(st.by), rep(st.bz), st.dx, st.dy, st.dz, st.gamma)


def _first(a, dims, axis):
    """Layer 0 along `axis` of a flat cell array."""
    nx, ny, nz = dims
    return np.take(a.reshape(-1, nz, ny, nx), [0], axis=3 - axis).reshape(a.shape[0], -1)


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("weights", ["js", "z"])
@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("na,nb", [(16, 8), (43, 3), (127, 1), (1, 129), (20, 13)])
def test_flat_axis_fluxes_and_step(precision, weights, axis, na, nb):
    from paper_1808_10633_gb300 import wombat as wb

    st = _flat_state(axis, na, nb, 17 * na + nb)
    out = []
    for n in (1, 2, 8):
        d = st if n == 1 else _deep(st, axis, n)
        with wb.Grid.from_state(d, precision=precision, weights=weights) as g:
            F = [_first(g.face_fluxes(a), d.dims, axis) for a in range(3)]
            g.step(1e-3, 1)
            U, b = g.get_state()
            out.append(F + [_first(U.reshape(8, -1), d.dims, axis), _first(b.reshape(3, -1), d.dims, axis)])
    for got in out[1:]:
        for x, y in zip(out[0], got):
            scale = np.maximum(np.abs(y).max(axis=1, keepdims=True), 1e-3 * np.abs(y).max())
            assert np.all(np.abs(x - y) <= 8 * EPS[precision] * scale)


def test_flat_patches_among_others_in_every_tile_table():
    """Patches with and without flat axes in one grid: each tile table gives
    the bits of the patches run on their own."""
    from paper_1808_10633_gb300 import inputs
    from paper_1808_10633_gb300 import wombat as wb

    dims = [(24, 20, 1), (1, 40, 17), (18, 19, 21), (65, 1, 3)]
    sts = [inputs.perturbed(*d, seed=5 + k, jump=True) for k, d in enumerate(dims)]
    for s in sts:
        s.dx = s.dy = s.dz = 1.0 / 32
    alone = []
    for s in sts:
        with wb.Grid.from_state(s, precision="fp32") as g:
            g.step(1e-3, 2)
            alone.append(g.get_state()[0])
    with wb.Grid.from_patches(sts, precision="fp32") as g:
        first = g.get_state()
        for c in range(len(wb.TILE_CANDIDATES)):
            g.set_tiles(c)
            g.set_state(*first)
            g.step(1e-3, 2)
            assert np.array_equal(g.get_state()[0], np.concatenate(alone)), c
