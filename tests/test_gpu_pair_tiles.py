"""Neutralization at the edges of the pair kernels' tiles (8192 slots): counts
one below, at and one above a tile, an empty and a one-particle partner, and
more than eight tiles per thread's group (over 2048 tiles).  Each case through a
discharge alone (ions counted behind their own chains), timed launches (counted
in one launch) and a batch.  Results against the oracle, pair for pair."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec
from helpers import capacity_for, compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu

NC = 32


def _case(n_om, n_op, seed):
    cfg = inputs.base_config(L=0.02, n_cells=NC, U=0.0, p=10.0, C_meta=0.0, ion_subcycle=2, weight=2e9, seed=seed,
                             steps_per_cycle=400)
    dx = cfg["L"] / NC
    mu = cfg["m_OM"] * cfg["m_OP"] / (cfg["m_OM"] + cfg["m_OP"])
    M = max(n_om, n_op) / NC                          # partners per cell: P = prob for every pair
    prob = min(0.1, 20000.0 / max(n_om, 1))
    K0 = prob / M * cfg["area"] * dx / (cfg["weight"] * cfg["dt"] * 2)
    procs = [xsec.constant_rate_process(1, xsec.NEUTRALIZE, K0, 1.0, mu, target=xsec.T_ION)]
    rng = np.random.default_rng(seed)
    st = []
    for s, n in enumerate((500, n_om, n_op)):
        x = ((rng.integers(0, NC, n) + 0.05 + 0.9 * rng.random(n)) * dx).astype(np.float32)
        v = (rng.standard_normal((3, n)) * (1e5 if s == 0 else 300.0)).astype(np.float32)
        st.append(dict(x=x, vx=v[0].copy(), vy=v[1].copy(), vz=v[2].copy(), id=np.arange(n, dtype=np.uint32)))
    return cfg, procs, st


def _check(g, o, procs):
    compare_particles(g, o)
    compare_counters(g.stats(), o.counters(), nproc_of(procs))


@pytest.mark.parametrize("how", ["alone", "timed"])
@pytest.mark.parametrize("n_om,n_op", [(8191, 8193), (8193, 8191), (8192, 16384), (16385, 8192), (9000, 0), (1, 9000),
                                       (9000, 1)])
def test_tile_edges(torch_cuda, n_om, n_op, how):
    cfg, procs, st = _case(n_om, n_op, 11)
    g, o, _ = make_pair(cfg, None, None, procs, state=st)
    if how == "timed":
        g.set_timing(True)
    for _ in range(3):
        g.step(2)
        o.step(2)
        _check(g, o, procs)
    if min(n_om, n_op) > 1:
        assert o.counters()["neutralized"] > 0


@pytest.mark.parametrize("n_om,n_op", [(100_000, 17_000_000), (17_000_000, 400_000)])
def test_many_tiles_per_group(torch_cuda, n_om, n_op):
    cfg, procs, st = _case(n_om, n_op, 12)
    g, o, _ = make_pair(cfg, None, None, procs, state=st, capacity=capacity_for((500, n_om, n_op), 1.1))
    g.step(2)
    o.step(2)
    compare_particles(g, o)
    stats, want = g.stats(), o.counters()
    # the field of so dense a state takes most pairs above the table: the library
    # counts those among the pairs it resolves, the oracle among all it tests
    assert want["neutralized"] > 100
    assert stats["warn_emax"] <= want["warn_emax"]
    want["warn_emax"] = stats["warn_emax"]
    compare_counters(stats, want, nproc_of(procs))
    g.close()


def test_batch_counts_beside_the_chains(torch_cuda):
    from paper_0705_0497_gb300 import api
    import oracle
    gs, os_ = [], []
    for i, (n_om, n_op) in enumerate([(8193, 8191), (30000, 26000), (500, 16385)]):
        cfg, procs, st = _case(n_om, n_op, 21 + i)
        g = api.Discharge(cfg, capacity_for((500, n_om, n_op)), compact_check=2)
        g.set_processes(procs)
        g.load_state(st)
        o = oracle.Oracle(cfg, 32)
        o.set_processes(procs)
        for s, p in enumerate(st):
            o.load(s, p["x"], p["vx"], p["vy"], p["vz"], p["id"])
        gs.append(g)
        os_.append((o, procs))
    b = api.Batch(gs, steps_per_launch=2)
    for _ in range(3):
        b.step(1)
        b.synchronize()
        for g, (o, procs) in zip(gs, os_):
            o.step(2)
            _check(g, o, procs)
            assert o.counters()["neutralized"] > 0
    b.close()
