"""The list of pair candidates when none, a few, many or all of a warp's
particles pass the first bound, with dead slots among them and a last tile that
ends inside a warp: neutralization against the oracle, pair for pair."""
import numpy as np
import pytest

from paper_0705_0497_gb300 import inputs, xsec
from helpers import compare_counters, compare_particles, make_pair, nproc_of

pytestmark = pytest.mark.gpu

NC = 32


# the share of the O- that pass the first bound is about NC times prob
@pytest.mark.parametrize("prob", [1e-5, 1e-3, 1e-2, 0.5])
@pytest.mark.parametrize("n_om,n_op", [(2 * 8192 + 777, 17_000), (130, 8192)])
def test_listed_candidates(torch_cuda, prob, n_om, n_op):
    cfg = inputs.base_config(L=0.02, n_cells=NC, U=0.0, p=10.0, C_meta=0.0, ion_subcycle=1, weight=1e3, seed=9,
                             steps_per_cycle=400)
    mu = cfg["m_OM"] * cfg["m_OP"] / (cfg["m_OM"] + cfg["m_OP"])
    K0 = prob / (max(n_om, n_op) / NC) * cfg["area"] * (cfg["L"] / NC) / (cfg["weight"] * cfg["dt"])
    procs = [xsec.constant_rate_process(1, xsec.NEUTRALIZE, K0, 1.0, mu, target=xsec.T_ION)]
    rng = np.random.default_rng(n_om)
    st = []
    for s, n in enumerate((500, n_om, n_op)):
        x = ((0.01 + 0.98 * rng.random(n)) * cfg["L"]).astype(np.float32)
        v = (rng.standard_normal((3, n)) * (1e5 if s == 0 else 300.0)).astype(np.float32)
        if s == 1:                          # a fifth of the O- leaves in the first step
            x[::5] = 1e-6 * cfg["L"]
            v[0, ::5] = -1.0e4
        st.append(dict(x=x, vx=v[0].copy(), vy=v[1].copy(), vz=v[2].copy(), id=np.arange(n, dtype=np.uint32)))
    g, o, _ = make_pair(cfg, None, None, procs, state=st, compact_check=100)
    for _ in range(3):
        g.step(1)
        o.step(1)
        compare_particles(g, o)
        compare_counters(g.stats(), o.counters(), nproc_of(procs))
    c = o.counters()
    assert c["absorbed_1_0"] >= n_om // 5
    assert c["neutralized"] > 0 or prob * min(n_om, n_op) < 10
