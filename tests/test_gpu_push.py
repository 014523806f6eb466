"""Edges of the particle kernel's rounds and counters against the oracle: many
particles of one block in one cell (the weight sum of a cell passes 2^32),
velocities whose current term needs more than 32 bits, and ranges that end
inside a round of 128, for warps with contiguous ranges and in turn."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec
from helpers import capacity_for, compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu


def _state(cfg, counts, fast, one_cell, seed=3):
    rng = np.random.default_rng(seed)
    dx = cfg["L"] / cfg["n_cells"]
    out = []
    for s, n in enumerate(counts):
        x = (dx * rng.uniform(0.98, 0.9999, n)) if one_cell else cfg["L"] * rng.random(n)
        v = rng.standard_normal((3, n)) * (1.0e6 if s == 0 else 1.0e3)
        if fast and s == 0:
            v[0, ::7] = 3.0e7 * np.sign(v[0, ::7])      # |256 v| above 2^31
        x = np.minimum(x, cfg["L"] * (1 - 1e-6)).astype(np.float32)
        out.append(dict(x=x, vx=v[0].astype(np.float32), vy=v[1].astype(np.float32), vz=v[2].astype(np.float32),
                        id=np.arange(n, dtype=np.uint32)))
    return out


@pytest.mark.parametrize("counts,shape,one_cell", [((140_003, 70_001, 140_003), (1, 1, 1), True),
                                                   ((257, 1, 127), (1, 2, 3), False),
                                                   ((5000, 4099, 12_345), (3, 2, 7), False)])
def test_push_edges_match_oracle(torch_cuda, counts, shape, one_cell):
    cfg, _, _, _ = inputs.workload("parity_128", n_cells=3 if one_cell else 128, weight=1.0e3, ion_subcycle=2)
    cfg["dt"] *= 1e-3 if one_cell else 1.0              # one cell: stay in it
    procs = xsec.oxygen_set()
    g, o, _ = make_pair(cfg, counts, None, procs, capacity=capacity_for(counts, 2.0, 64),
                        state=_state(cfg, counts, True, one_cell))
    g.set_launch_shape(shape)
    g.step(5)
    o.step(5)
    compare_particles(g, o)
    compare_counters(g.stats(), o.counters(), nproc_of(procs))
    assert np.array_equal(g.charge()[0], o.charge()[0])
    J, sums = g.currents(0, 5), o.current_sums(0, 5)
    unit = inputs.QE * cfg["weight"] / (256.0 * cfg["area"] * cfg["L"])
    want = np.asarray(sums, np.float64).reshape(5, 3) * unit * np.array([-1.0, -1.0, 1.0])
    assert np.allclose(J[:, :3], want, rtol=1e-14, atol=0)
