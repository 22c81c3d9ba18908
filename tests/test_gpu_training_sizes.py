"""Loss, gradient and minibatch loss of the training kernels at the sizes where
their work splits: one record, a chunk of 32 less or more one, the last chunk
of the last block (43 blocks of 32 records) less or more one, an empty field.

Tolerances: the FP32 forward and backward pass of a record rounds about a
hundred times, 100 x 2^-24 = 6e-6 of each entry's typical product; the mean
over n random records may cancel to 1/sqrt(n) of that (n <= 1 400: 40 times),
so the gradient is compared to 3e-4 of its largest entry, and the loss (a sum
of non-negative terms) to 1e-5."""
import numpy as np
import pytest

from test_gpu_learned import _records

pytestmark = pytest.mark.gpu

LAM = 1e-2


def _case(counts, seed):
    rec = _records(7 * max(counts) + 8, seed)
    rec[:, 11] = 0
    out = []
    for f, n in enumerate(counts):
        r = rec[f::7][:n].copy()
        r[:, 0] = f
        out.append(r)
    flagged = rec[:5].copy()
    flagged[:, 11] = 1
    all_ = np.concatenate(out + [flagged])
    return all_[np.random.default_rng(seed).permutation(len(all_))]


def _params(seed):
    from oracle import learned as Lr

    return (np.random.default_rng(seed).standard_normal((7, Lr.NPARAM)) * 0.3).astype(np.float32)


@pytest.mark.parametrize("counts", [(1, 2, 31, 32, 33, 0, 64), (43 * 32 - 1, 43 * 32, 43 * 32 + 1, 1, 0, 44, 1000)])
def test_full_batch_gradient(counts):
    from oracle import learned as Lr
    from paper_1808_10633_gb300 import wombat as wb

    rec, par = _case(counts, 11), _params(12)
    loss, grad = wb.mlp_loss_grad(rec, par, LAM)
    again = wb.mlp_loss_grad(rec, par, LAM)
    assert np.array_equal(loss, again[0]) and np.array_equal(grad, again[1])
    for f, n in enumerate(counts):
        if n == 0:
            assert loss[f] == 0 and not grad[f].any()
            continue
        r = rec[(rec[:, 0] == f) & (rec[:, 11] == 0)].astype(np.float64)
        L, g = Lr.loss_and_grad(par[f].astype(np.float64), r[:, 1:7], r[:, 7:10], r[:, 10], LAM)
        assert loss[f] == pytest.approx(L, rel=1e-5), f
        assert np.abs(grad[f] - g).max() <= 3e-4 * np.abs(g).max(), f


@pytest.mark.parametrize("batch", [1, 31, 33, 43 * 32 + 1, 4097])
def test_minibatch_loss(batch):
    from oracle import learned as Lr
    from paper_1808_10633_gb300 import wombat as wb

    counts, seed = (50, 3, 200, 1, 0, 33, 700), 77
    rec, par = _case(counts, 13), _params(14)
    new, hist = wb.mlp_train(rec, par, 1, batch=batch, lr=1e-3, lam=LAM, seed=seed)

    def mix(z):
        with np.errstate(over="ignore"):
            z = z + np.uint64(0x9E3779B97F4A7C15)
            z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
            z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
            return z ^ (z >> np.uint64(31))

    slots = np.arange(batch, dtype=np.uint64)
    for f, n in enumerate(counts):
        if n == 0:
            assert hist[0, f] == 0 and np.array_equal(new[f], par[f])
            continue
        r = rec[(rec[:, 0] == f) & (rec[:, 11] == 0)].astype(np.float64)
        pick = (mix(np.uint64(seed) ^ mix(np.uint64(f * 8191) + slots)) % np.uint64(n)).astype(int)
        L, g = Lr.loss_and_grad(par[f].astype(np.float64), r[pick, 1:7], r[pick, 7:10], r[pick, 10], LAM)
        assert hist[0, f] == pytest.approx(L, rel=1e-5), f
        # Adam's first step moves each parameter by lr against its gradient's sign
        big = np.abs(g) > 1e-3 * np.abs(g).max()
        assert np.allclose((new[f] - par[f])[big], -1e-3 * np.sign(g[big]), rtol=1e-2, atol=1e-7), f
