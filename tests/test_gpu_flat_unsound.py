"""Sweeps along an axis of one cell, one thread per cell, against the interface
arithmetic on the same grid linked to itself: cells without an eigen-structure (no
positive density or pressure, infinite or NaN entries) give NaN fluxes on both, the
others the same to 8 ulp of a component's scale (a handful of roundings)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

EPS = {"fp64": 2.0 ** -52, "fp32": 2.0 ** -23}


@pytest.mark.parametrize("precision", ["fp64", "fp32"])
@pytest.mark.parametrize("weights", ["js", "z"])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_cells_without_an_eigen_structure(precision, weights, axis):
    from paper_1808_10633_gb300 import bricks, inputs
    from paper_1808_10633_gb300 import wombat as wb

    dims = [13, 11, 9]
    dims[axis] = 1
    st = inputs.perturbed(*dims, seed=axis)
    flat = [st.U[k].reshape(-1) for k in range(8)]
    for cell, field, value in ((3, 7, 1e-3), (10, 0, -1.0), (21, 0, 0.0), (33, 7, -2.0), (40, 7, np.inf), (52, 1, np.nan),
                               (61, 2, np.inf), (70, 0, np.inf)):
        flat[field][cell] = value
    cuts = tuple([0, n] for n in dims)
    kw = dict(precision=precision, weights=weights)
    with wb.Grid.from_state(st, **kw) as g:
        F = g.face_fluxes(axis)
    with wb.Grid.from_bricks(st, cuts, **kw) as g:
        G = g.face_fluxes(axis)
    assert np.array_equal(np.isnan(F), np.isnan(G)), (np.argwhere(np.isnan(F[0])), np.argwhere(np.isnan(G[0])))
    good = ~np.isnan(G[0])
    assert 0 < (~good).sum() <= 8 and np.isfinite(G[:, good]).all()
    scale = np.maximum(np.abs(G[:, good]).max(axis=1, keepdims=True), 1e-3 * np.abs(G[:, good]).max())
    assert np.all(np.abs(F - G)[:, good] <= 8 * EPS[precision] * scale)
