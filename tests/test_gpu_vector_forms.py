"""FP32 and FP64 grids above the limit of the one-launch stage whose patches' x extents
are multiples of the vector width take the vector forms of the EMF and update kernels:
the bits of the patch on its own, both EMF modes and integrators."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,filler", [("fp32", 60), ("fp64", 44)])
@pytest.mark.parametrize("integrator", ["ssprk3", "rk4"])
@pytest.mark.parametrize("emf_mode", [0, 1])
@pytest.mark.parametrize("dims", [(24, 20, 16), (4, 3, 5), (36, 9, 1), (8, 1, 12), (260, 2, 2)])
def test_vector_forms_give_the_same_bits(precision, filler, integrator, emf_mode, dims):
    from paper_1808_10633_gb300 import inputs
    from paper_1808_10633_gb300 import wombat as wb

    st = inputs.perturbed(*dims, seed=9, jump=True)
    st.dx = st.dy = st.dz = 1 / 32
    kw = dict(precision=precision, integrator=integrator, emf_mode=emf_mode)
    fill = inputs.uniform(filler, filler, filler, dx=1 / 32, dy=1 / 32, dz=1 / 32)
    n = st.bx.size
    with wb.Grid.from_state(st, **kw) as g:
        g.step(1e-3, 2)
        U, b = g.get_state()
    with wb.Grid.from_patches([st, fill], **kw) as g:
        g.step(1e-3, 2)
        V, c = g.get_state()
    assert np.array_equal(U, V[:8 * n]) and np.array_equal(b, c[:3 * n])
