"""The autotuner's first and last candidate are one table: one time for both."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp32", "fp64"])
def test_one_table_has_one_time(precision):
    from paper_1808_10633_gb300 import inputs
    from paper_1808_10633_gb300 import wombat as wb

    with wb.Grid.from_state(inputs.perturbed(33, 20, 17, seed=1), precision=precision) as g:
        for _ in range(3):
            ms = g.autotune()
            assert ms.shape == (3, 5) and np.all(ms > 0) and np.array_equal(ms[:, 0], ms[:, 4])
