"""Sums over records in the training kernels are FP64: losses whose sum leaves the FP32
range, in one chunk of 32 records, over the blocks, and in a minibatch, have a finite
mean.  Tolerance: the loss of a record is a square of an FP32 difference, three
roundings, and all are positive: 4 x 2^-24."""
import numpy as np
import pytest

from test_gpu_learned import _records

pytestmark = pytest.mark.gpu


def _case(n, size):
    rec = _records(7 * n, 21)
    rec[:, 11] = 0
    rec[:, 10] = size * np.random.default_rng(n).uniform(1, 2, len(rec)) * np.sign(rec[:, 10] + 0.5)
    par = (np.random.default_rng(3).standard_normal((7, 1379)) * 0.3).astype(np.float32)
    # the output is of order one: the loss is the target squared to 1e-17
    want = [np.mean(rec[rec[:, 0] == f, 10].astype(np.float64) ** 2) for f in range(7)]
    return rec, par, np.array(want)


@pytest.mark.parametrize("n,size", [(32, 4e18), (300, 1.2e18), (3000, 8e17)])
def test_sums_beyond_the_fp32_range(n, size):
    from paper_1808_10633_gb300 import wombat as wb

    rec, par, want = _case(n, size)
    assert np.all(want * n > 3.5e38)
    loss, grad = wb.mlp_loss_grad(rec, par, 0.0)
    assert np.all(np.abs(loss / want - 1) <= 4 * 2.0 ** -24), loss / want
    assert np.isfinite(grad).all() and np.abs(grad).max() > 0
    new, hist = wb.mlp_train(rec, par, 1, batch=4 * n, lr=1e-3, lam=0.0, seed=5)
    assert np.isfinite(hist).all() and np.isfinite(new).all()
    assert np.all(np.abs(hist[0] / want - 1) < 0.5), hist[0] / want
