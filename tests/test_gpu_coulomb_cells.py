"""The Coulomb cell sort at the cell counts where its scatter changes blocks,
and with cells of no, one and many particles, against the oracle."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec
from helpers import compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nc,counts", [(1, (700, 3, 1)), (4096, (9000, 8192, 8193)), (4097, (9000, 100, 20_000)),
                                       (8192, (16_385, 5000, 3))])
def test_coulomb_cell_counts(torch_cuda, Nc, counts):
    cfg = inputs.base_config(L=0.02, n_cells=Nc, U=50.0, p=10.0, C_meta=0.0, ion_subcycle=1, weight=1e9, seed=4,
                             steps_per_cycle=4000)
    procs = xsec.oxygen_set()
    rng = np.random.default_rng(Nc)
    st = []
    for s, n in enumerate(counts):
        x = (rng.random(n) ** 3 * 0.9 * cfg["L"]).astype(np.float32)      # crowded and empty cells
        v = (rng.standard_normal((3, n)) * (1.0e6 if s == 0 else 500.0)).astype(np.float32)
        st.append(dict(x=x, vx=v[0].copy(), vy=v[1].copy(), vz=v[2].copy(), id=np.arange(n, dtype=np.uint32)))
    g, o, _ = make_pair(cfg, None, None, procs, state=st)
    g.set_coulomb(63, 10.0)
    o.set_coulomb(63, 10.0)
    g.step(3)
    o.step(3)
    compare_particles(g, o)
    compare_counters(g.stats(), o.counters(), nproc_of(procs))
    assert o.counters()["coulomb_pairs"] > 300
