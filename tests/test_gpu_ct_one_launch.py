"""Small grids take the EMFs and the update of a stage in one launch; the same
patch in a grid above the limit takes two.  Both share their arithmetic with
explicit rounding, so the patch's bits must agree: periodic and linked patches,
odd and thin extents, both EMF modes, both integrators."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

LIMIT = {"fp32": 180_000, "fp64": 80_000}


def _filler(n):
    from paper_1808_10633_gb300 import inputs

    return inputs.uniform(n, n, n, dx=1 / 32, dy=1 / 32, dz=1 / 32)


@pytest.mark.parametrize("precision,filler", [("fp32", 58), ("fp64", 44)])
@pytest.mark.parametrize("integrator", ["ssprk3", "rk4"])
@pytest.mark.parametrize("emf_mode", [0, 1])
@pytest.mark.parametrize("dims", [(24, 20, 16), (7, 3, 5), (33, 9, 1), (1, 1, 12), (2, 2, 2)])
def test_one_launch_equals_two(precision, filler, integrator, emf_mode, dims):
    from paper_1808_10633_gb300 import inputs
    from paper_1808_10633_gb300 import wombat as wb

    st = inputs.perturbed(*dims, seed=3, jump=dims[0] > 4)
    st.dx = st.dy = st.dz = 1 / 32
    kw = dict(precision=precision, integrator=integrator, emf_mode=emf_mode)
    n = st.bx.size
    assert n <= LIMIT[precision] < n + filler ** 3
    with wb.Grid.from_state(st, **kw) as g:
        g.step(1e-3, 2)
        U, b = g.get_state()
    with wb.Grid.from_patches([st, _filler(filler)], **kw) as g:
        g.step(1e-3, 2)
        V, c = g.get_state()
    assert np.array_equal(U, V[:8 * n]) and np.array_equal(b, c[:3 * n])


@pytest.mark.parametrize("precision,filler", [("fp32", 58), ("fp64", 44)])
def test_one_launch_equals_two_on_linked_bricks(precision, filler):
    from paper_1808_10633_gb300 import bricks, inputs
    from paper_1808_10633_gb300 import wombat as wb

    st = inputs.perturbed(19, 16, 14, seed=8, jump=True)
    st.dx = st.dy = st.dz = 1 / 32
    cuts = ([0, 8, 19], [0, 5, 16], [0, 3, 9, 14])
    fl = _filler(filler)
    dims, links = bricks.brick_dims(cuts), bricks.brick_links(cuts)
    U0, b0 = bricks.split(st.U, np.stack([st.bx, st.by, st.bz]), cuts)
    own = np.full(27, len(dims), dtype=np.int32)      # the filler is periodic on itself
    n = st.bx.size
    with wb.Grid(dims, 1 / 32, 1 / 32, 1 / 32, U0, b0, precision=precision, links=links) as g:
        g.step(1e-3, 2)
        U, b = g.get_state()
    with wb.Grid(dims + [fl.dims], 1 / 32, 1 / 32, 1 / 32, np.concatenate([U0, fl.U.ravel()]),
                 np.concatenate([b0, np.stack([fl.bx, fl.by, fl.bz]).ravel()]), precision=precision,
                 links=np.concatenate([links, own])) as g:
        g.step(1e-3, 2)
        V, c = g.get_state()
    assert np.array_equal(U, V[:8 * n]) and np.array_equal(b, c[:3 * n])
