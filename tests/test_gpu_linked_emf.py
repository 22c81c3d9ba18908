"""EMFs of linked FP32 bricks in a grid large enough for the EMF kernel of its
own: cells inside a brick reach their neighbours at fixed distances, those at its
lower faces, edges and corner through the links.  The shared arithmetic is
explicitly rounded, so the bricks must give the bits of the uncut world: thin and
uneven bricks, both EMF modes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("emf_mode", [0, 1])
@pytest.mark.parametrize("dims,cuts", [
    ((67, 59, 53), ([0, 3, 40, 67], [0, 29, 59], [0, 4, 8, 53])),
    ((64, 57, 56), ([0, 64], [0, 3, 6, 57], [0, 33, 56])),
    ((61, 3, 1000), ([0, 32, 61], [0, 3], [0, 997, 1000])),
])
def test_large_linked_bricks_equal_the_uncut_world(dims, cuts, emf_mode):
    from paper_1808_10633_gb300 import bricks, inputs
    from paper_1808_10633_gb300 import wombat as wb

    st = inputs.perturbed(*dims, seed=12, jump=True)
    st.dx = st.dy = st.dz = 1 / 64
    kw = dict(precision="fp32", emf_mode=emf_mode)
    assert st.bx.size > 180_000
    with wb.Grid.from_state(st, **kw) as g:
        g.step(5e-4, 2)
        U, b = g.get_state()
    with wb.Grid.from_bricks(st, cuts, **kw) as g:
        g.step(5e-4, 2)
        V, c = g.get_state()
    V, c = bricks.join(V, c, cuts)
    assert np.array_equal(U.ravel(), V.ravel()) and np.array_equal(b.ravel(), c.ravel())
