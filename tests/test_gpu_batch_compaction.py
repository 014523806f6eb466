"""Compaction in a batch whose compaction launch has far more blocks than the
GPU runs at once (many discharges, capacities far above the particle counts):
blocks still start while others commit their discharge's new slot counts.  Each
discharge must give what it gives alone."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("branches", [False, True])
def test_compaction_in_a_large_batch(torch_cuda, monkeypatch, branches):
    from paper_0705_0497_gb300 import api
    if branches:
        monkeypatch.setenv("O2PIC_BATCH_BRANCHES", "1")
    procs = xsec.oxygen_set()

    def make(cfg, counts, T):
        g = api.Discharge(cfg, tuple(300_000 for _ in counts), compact_check=10)
        g.set_processes(procs)
        st = inputs.initial_state(cfg, counts, T)
        st[0]["vx"] *= np.float32(4.0)          # electrons lost to the walls from the first steps on
        g.load_state(st)
        return g

    sweep = [(c, (n[0] + 9000, n[1], n[2]), T) for c, n, T in inputs.batch_sweep(40, seed=3, scale=0.01)]
    ds = [make(*s) for s in sweep]
    b = api.Batch(ds, steps_per_launch=20)
    b.step(15)
    b.synchronize()
    for i in (0, 17, 39):
        alone = make(*sweep[i])
        alone.step(300)
        sa, sb = alone.stats(), ds[i].stats()
        assert sa == sb
        assert sa["slots_0"] < sweep[i][1][0] + sa["born_0"]      # compacted at least once
        for s in range(3):
            p, q = alone.particles(s, flight=True), ds[i].particles(s, flight=True)
            for k in p:
                assert np.array_equal(p[k], q[k]), (i, s, k)
        alone.close()
    b.close()
