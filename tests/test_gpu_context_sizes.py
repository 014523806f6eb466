"""Discharges of very different cell counts side by side: creating a small one
leaves the kernels' shared-memory limits of a larger one as they were, alone
and in a batch with it, and the launch shape chosen for a larger one does not
depend on what was created before."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import api, inputs, xsec
from helpers import compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("large", [8192, 2048])
def test_larger_discharge_after_a_smaller_one(torch_cuda, large):
    procs = xsec.oxygen_set()
    counts = (3000, 1000, 3500)

    def make(Nc):
        cfg, _, T, _ = inputs.workload("parity_128", n_cells=Nc, ion_subcycle=2)
        return make_pair(cfg, counts, T, procs, compact_check=2)[:2]

    def check(g, o):
        compare_particles(g, o)
        compare_counters(g.stats(), o.counters(), nproc_of(procs))
        assert np.array_equal(g.charge()[0], o.charge()[0])

    a, oa = make(large)
    shape = a.launch_shape()
    b, ob = make(32)
    a.step(4)
    oa.step(4)
    check(a, oa)
    b.step(4)
    ob.step(4)
    check(b, ob)
    a.set_processes(procs)
    assert a.launch_shape() == shape
    oa.set_processes(procs)
    batch = api.Batch([a, b], steps_per_launch=4)
    batch.step(2)
    batch.synchronize()
    for g, o in ((a, oa), (b, ob)):
        o.step(8)
        check(g, o)
    batch.close()
    a.close()
    b.close()
