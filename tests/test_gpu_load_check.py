"""The check of loaded particles at the edges of its blocks: the largest id
(wherever it is) sets the next id, and one bad value anywhere refuses the load."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import api, inputs

pytestmark = pytest.mark.gpu

ROUND = 8 * 152 * 256      # particles of one pass of the whole grid


@pytest.mark.parametrize("n", [1, 31, 33, 255, 256, 257, ROUND - 1, ROUND, ROUND + 1, 2 * ROUND + 300])
def test_largest_id_and_bad_values(torch_cuda, n):
    cfg, _, _, _ = inputs.workload("parity_128")
    g = api.Discharge(cfg, (n + 16, 100, 100))
    x = np.full(n, 0.5 * cfg["L"], np.float32)
    z = np.zeros(n, np.float32)
    ids = np.arange(n, dtype=np.uint32)
    for at in {0, n // 2, n - 1}:
        big = ids.copy()
        big[at] = 3_000_000_000
        g.load(0, x, z, z, z, big)
        with pytest.raises(api.O2picError):
            g.set_next_id(0, 3_000_000_000)
        g.set_next_id(0, 3_000_000_001)
        for k in range(4):
            a = [x.copy(), z.copy(), z.copy(), z.copy()]
            a[k][at] = (np.nan, np.inf, -np.inf, np.nan)[k]
            with pytest.raises(api.O2picError) as e:
                g.load(0, *a, ids)
            assert e.value.code == -1 and g.count(0) == 0
    g.load(0, x, z, z, z, ids)
    assert g.count(0) == n
    g.set_next_id(0, n)
    g.close()
