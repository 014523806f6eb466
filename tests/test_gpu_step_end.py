"""The end-of-step kernel's cluster of blocks at cell counts around its shares
(fewer nodes than blocks, one more and one less than a multiple of a block's
threads) and the ion kernel with more collisions of a warp than it has lanes,
against the oracle."""
import math

import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec
from helpers import compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("Nc", [1, 2, 7, 8, 255, 257, 2047, 2049, 4096])
def test_field_at_share_edges(torch_cuda, Nc):
    import oracle
    cfg, _, T, _ = inputs.workload("parity_128", n_cells=Nc, ion_subcycle=2)
    procs = xsec.oxygen_set()
    g, o, _ = make_pair(cfg, (3000, 1000, 3500), T, procs)
    for chunk in (1, 8):
        g.step(chunk)
        o.step(chunk)
        compare_particles(g, o)
        compare_counters(g.stats(), o.counters(), nproc_of(procs))
        for a, b in zip(g.charge(), o.charge()):
            assert np.array_equal(a, b)
    Q = g.charge()[0].astype(np.int64)
    V0 = cfg["U"] * math.sin(2.0 * math.pi * cfg["f"] * (g.stats()["step"] * cfg["dt"]))
    phi64, E64 = oracle.solve_field(Nc, cfg["L"] / Nc, cfg["weight"], cfg["area"], V0, Q[2] - Q[0] - Q[1])
    phi, E = g.field()
    assert np.array_equal(E, E64.astype(np.float32))
    assert np.array_equal(phi, phi64)


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5)])
def test_many_collisions_per_warp(torch_cuda, shape):
    cfg, _, T, _ = inputs.workload("parity_128", p=2.0e4, ion_subcycle=2)
    procs = xsec.oxygen_set()
    counts = (2000, 9000, 9000)
    g, o, _ = make_pair(cfg, counts, T, procs)
    g.set_launch_shape(shape)
    g.step(6)
    o.step(6)
    compare_particles(g, o)
    c = o.counters()
    compare_counters(g.stats(), c, nproc_of(procs))
