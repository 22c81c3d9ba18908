"""State copies to page-locked arrays in place and to pageable ones through device
staging take different kernels: the same bits, for linked bricks and uneven patches,
with and without each of the two arrays."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def _grid(links, precision):
    from paper_1808_10633_gb300 import inputs
    from paper_1808_10633_gb300 import wombat as wb

    if links:
        st = inputs.perturbed(23, 14, 11, seed=4, jump=True)
        return wb.Grid.from_bricks(st, ([0, 9, 23], [0, 3, 14], [0, 11]), precision=precision)
    sts = [inputs.perturbed(*d, seed=k) for k, d in enumerate([(5, 7, 9), (40, 1, 3), (16, 16, 2)])]
    for s in sts:
        s.dx = s.dy = s.dz = 0.1
    return wb.Grid.from_patches(sts, precision=precision)


@pytest.mark.parametrize("links", [False, True])
@pytest.mark.parametrize("precision,dtype", [("fp32", torch.float32), ("fp32", torch.float64), ("fp64", torch.float64)])
def test_pinned_and_pageable_copies_agree(links, precision, dtype):
    from paper_1808_10633_gb300 import wombat as wb

    with _grid(links, precision) as g:
        N = g.ncells
        get = g._lib.wb_get_state_f32 if dtype == torch.float32 else g._lib.wb_get_state
        outs = []
        for pinned in (True, False):
            for want in ((1, 1), (1, 0), (0, 1)):
                U, b = (torch.full((n * N,), -7.0, dtype=dtype, pin_memory=pinned) for n in (8, 3))
                rc = get(g._h, *(ctypes.c_void_p(t.data_ptr()) if w else None for t, w in zip((U, b), want)))
                assert rc == wb.WB_OK
                for t, w in zip((U, b), want):
                    assert bool((t == -7).any()) != bool(w)
                outs.append((U, b, want))
        for U, b, want in outs[1:]:
            for t, ref, w in zip((U, b), outs[0], want):
                assert not w or torch.equal(t, ref)
        U, b = outs[0][:2]
        back = []
        for pinned in (True, False):
            V, c = 2 * U, 2 * b
            if pinned:
                V, c = V.pin_memory(), c.pin_memory()
                g.set_state(V, c)
            else:
                g.set_state(V.numpy(), c.numpy())
            back.append(g.get_state())
        assert all(np.array_equal(p, q) for p, q in zip(*back))
        assert np.array_equal(back[0][1], 2 * b.numpy())
