"""What lies in the collision records' memory after a step's collisions: the
candidates of (16) and (17) and the cell sort of the Coulomb collisions.  Every
particle is a candidate, many collide and react, and the arrays have no slot to
spare, so any overlap would change results; all of them against the oracle."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec
from helpers import compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu

NC = 32
N2 = 1.0e20        # gas density of the test collisions, m^-3


def _rate(prob, dt):
    return -np.log(1.0 - prob) / dt


@pytest.mark.parametrize("coulomb", [0, 63])
@pytest.mark.parametrize("rec", [False, True])
@pytest.mark.parametrize("counts", [(3343, 9001, 12_345), (129, 8193, 8321)])
def test_lists_share_the_records(torch_cuda, counts, rec, coulomb):
    cfg = inputs.base_config(L=0.02, n_cells=NC, U=0.0, p=10.0, C_meta=0.0, ion_subcycle=2, weight=2e9, seed=7,
                             steps_per_cycle=400)
    dt, dti = cfg["dt"], 2 * cfg["dt"]
    cfg["p"] = N2 * 1.380649e-23 * cfg["T_gas"]
    mass = [inputs.species_mass(cfg, s) for s in range(3)]
    red = lambda a, b: a * b / (a + b)  # noqa: E731
    procs = [xsec.constant_rate_process(0, xsec.ELASTIC, _rate(0.5, dt), N2, mass[0])]
    procs += [xsec.constant_rate_process(s, xsec.ELASTIC, _rate(0.5, dti), N2, red(mass[s], cfg["M_gas"])) for s in (1, 2)]
    pair = lambda prob, n: prob / (n / NC) * cfg["area"] * (cfg["L"] / NC) / (cfg["weight"] * dti)  # noqa: E731
    procs.append(xsec.constant_rate_process(1, xsec.NEUTRALIZE, pair(0.05, counts[2]), 1.0, red(mass[1], mass[2]),
                                            target=xsec.T_ION))
    if rec:
        procs.append(xsec.constant_rate_process(0, xsec.RECOMBINE, pair(0.05, counts[2]), 1.0, red(mass[0], mass[2]),
                                                target=xsec.T_ION))
    rng = np.random.default_rng(5)
    st = []
    for s, n in enumerate(counts):
        x = ((0.01 + 0.98 * rng.random(n)) * cfg["L"]).astype(np.float32)
        v = (rng.standard_normal((3, n)) * (2e5 if s == 0 else 300.0)).astype(np.float32)
        st.append(dict(x=x, vx=v[0].copy(), vy=v[1].copy(), vz=v[2].copy(), id=np.arange(n, dtype=np.uint32)))
    g, o, _ = make_pair(cfg, None, None, procs, state=st, capacity=counts)
    if coulomb:
        g.set_coulomb(coulomb)
        o.set_coulomb(coulomb, 10.0)
    for _ in range(3):
        g.step(2)
        o.step(2)
        compare_particles(g, o)
        compare_counters(g.stats(), o.counters(), nproc_of(procs))
    c = o.counters()
    assert c["neutralized"] > 500 and (not rec or c["recombined"] > 5)
    assert min(c["events_0_0"] / counts[0], c["events_1_0"] / counts[1], c["events_2_0"] / counts[2]) > 0.5
