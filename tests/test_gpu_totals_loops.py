"""FP32 totals where a thread's loop runs many times: all values of a field lie in the
cells one thread adds (every 256th of a block's chunk of a 1024th of the cells), the
rest is zero.

The errors of its FP32 additions are kept to 2^-72 of the sum and joined with it in
FP64, two roundings: 2 x 2^-53 of the magnitudes.  Values that leave the FP32 range on
the way are added in FP64, one rounding each."""
import math

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("per", [3, 24, 64, 200])
@pytest.mark.parametrize("kind", [0, 20, 40, "huge"])
def test_one_thread_adds_many_values(per, kind):
    import torch

    from paper_1808_10633_gb300 import wombat as wb

    n = per * 1024 * 256 + 77
    chunk = -(-n // 1024)
    rng = np.random.default_rng(per)
    d = torch.zeros((8, n), dtype=torch.float32, device="cuda")
    x = rng.standard_normal((8, per))
    if kind == "huge":
        x = np.where(x < 0, -3.3e38, 3.2e38) * rng.uniform(0.9, 1.0, x.shape)
    else:
        x *= np.exp2(rng.uniform(-kind, 0, x.shape))
    x = x.astype(np.float32)
    for f in range(8):                       # field f: thread 5 f of block 100 f
        d[f, 100 * f * chunk + 5 * f + 256 * torch.arange(per)] = torch.from_numpy(x[f]).cuda()
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    wb.conserved_totals_noalloc(d.data_ptr(), "fp32", n, 1.0, out.data_ptr(),
                                torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    got = out.cpu().numpy()[[0, 1, 2, 3, 7, 4, 5, 6]]
    roundings = per if kind == "huge" else 2
    for f in range(8):
        v = x[f].astype(np.float64)
        assert abs(got[f] - math.fsum(v)) <= roundings * 2.0 ** -53 * math.fsum(np.abs(v)), f
