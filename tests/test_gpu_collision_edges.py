"""Collisions at the edges of their counters and lists against the oracle: a
cell's weight sum that falls below zero (modulo 2^32) when an attached electron
leaves it, and warps whose real collisions fill their lanes several times over
before what is left is pooled."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec
from helpers import compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu

N2 = 1.0e20        # gas density, m^-3


def _config(**kw):
    cfg = inputs.base_config(U=0.0, p=N2 * 1.380649e-23 * 300.0, C_meta=0.0, steps_per_cycle=400, **kw)
    assert cfg["T_gas"] == 300.0
    return cfg


def _rate(prob, dt):
    return -np.log(1.0 - prob) / dt


def test_weight_sum_borrows(torch_cuda):
    # 2^17 electrons at rest in x at a cell's centre (weight 2^15 each): the
    # block's sum is 2^32, its 32-bit counter 0, when the first one is attached
    n = 1 << 17
    cfg = _config(L=2.0 ** -5, n_cells=4, ion_subcycle=2, weight=0.0, seed=3)
    procs = [xsec.constant_rate_process(0, xsec.ATTACH, _rate(0.3, cfg["dt"]), N2, cfg["m_e"])]
    st = []
    for s, m in enumerate((n, 10, 10)):
        z = np.zeros(m, np.float32)
        st.append(dict(x=np.full(m, 1.5 * 2.0 ** -7, np.float32), vx=z, vy=z + 1.0e6, vz=z,
                       id=np.arange(m, dtype=np.uint32)))
    g, o, _ = make_pair(cfg, None, None, procs, state=st, capacity=(2 * n, 2 * n, 64))
    g.set_launch_shape((1, 1, 1))
    for _ in range(2):
        g.step(1)
        o.step(1)
        compare_particles(g, o)
        compare_counters(g.stats(), o.counters(), nproc_of(procs))
        for a, b in zip(g.charge(), o.charge()):
            assert np.array_equal(a, b)
    assert o.counters()["events_0_0"] > n // 4


@pytest.mark.parametrize("shape", [(1, 1, 1), (2, 3, 5)])
def test_full_lanes_of_collisions(torch_cuda, shape):
    cfg = _config(L=0.02, n_cells=64, ion_subcycle=2, weight=1.0e3, seed=6)
    dt, dti = cfg["dt"], 2 * cfg["dt"]
    m = [inputs.species_mass(cfg, s) for s in range(3)]
    mu = [m[0]] + [a * cfg["M_gas"] / (a + cfg["M_gas"]) for a in m[1:]]
    procs = [xsec.constant_rate_process(0, xsec.ELASTIC, _rate(0.4, dt), N2, mu[0]),
             xsec.constant_rate_process(0, xsec.ATTACH, _rate(0.1, dt), N2, mu[0]),
             xsec.constant_rate_process(1, xsec.ELASTIC, _rate(0.4, dti), N2, mu[1]),
             xsec.constant_rate_process(1, xsec.DETACH, _rate(0.1, dti), N2, mu[1]),
             xsec.constant_rate_process(2, xsec.CX, _rate(0.4, dti), N2, mu[2]),
             xsec.constant_rate_process(2, xsec.ELASTIC, _rate(0.1, dti), N2, mu[2])]
    counts = (9000, 9000, 9000)
    rng = np.random.default_rng(8)
    st = []
    for s, n in enumerate(counts):
        x = (rng.random(n) * 0.999 * cfg["L"]).astype(np.float32)
        v = (rng.standard_normal((3, n)) * (1.0e6 if s == 0 else 300.0)).astype(np.float32)
        st.append(dict(x=x, vx=v[0].copy(), vy=v[1].copy(), vz=v[2].copy(), id=np.arange(n, dtype=np.uint32)))
    g, o, _ = make_pair(cfg, None, None, procs, state=st)
    g.set_launch_shape(shape)
    steps = 4
    g.step(steps)
    o.step(steps)
    compare_particles(g, o)
    c = o.counters()
    compare_counters(g.stats(), c, nproc_of(procs))
    assert np.array_equal(g.charge()[0], o.charge()[0])
    for s, pushes in enumerate((steps, steps // 2, steps // 2)):
        per_warp = (c[f"events_{s}_0"] + c[f"events_{s}_1"]) / pushes / (8 * shape[s])
        assert per_warp > 64, (s, per_warp)
