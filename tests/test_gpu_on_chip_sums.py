"""The inner products of the solve held on the chip are FP64 from the warps'
partials on. A problem scaled so that every partial fits FP32 and their total
does not (1e39; at least 150 warps hold it) is solved like the unscaled one: the
equations are linear, so the two differ by twice the precision's bar at most."""
import numpy as np
import pytest

import workloads as W
from oracle import transient

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,bar", [("fp32_refined", 1e-8), ("fp32_plain", 1e-4)])
@pytest.mark.parametrize("element", ["q1", "p1"])
def test_a_total_beyond_fp32(element, precision, bar):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(48, 44, 46, seed=8, dirichlet={4: 0.0}, theta=0.5, dt=0.01, nsteps=1, contrast=(0.1, 10.0),
                     rtol=1e-10 if precision == "fp32_refined" else 1e-6)
    p.element = element
    u0 = W.apply_dirichlet_values(p, np.random.default_rng(9).standard_normal(p.n_nodes))
    S = transient.build_system(p)
    free = np.ones(p.n_nodes, dtype=bool)
    free[np.isfinite(W.apply_dirichlet_values(p, np.full(p.n_nodes, np.nan)))] = False
    r = np.where(free, -(S.K @ u0), 0.0)  # b - A u0 without loads
    delta = float(np.sum(r * r / (S.M.diagonal() / p.dt + p.theta * S.K.diagonal())))
    scale = np.sqrt(1e39 / delta)
    got = []
    for f in (1.0, scale):
        with hg.Simulation.from_problem(p, precision=precision) as s:
            hg.heat_set_state(s.sim, f * u0, p.n_nodes)
            rc, st = hg.heat_step_nocheck(s.sim, 1)
            assert rc == 0, (f, hg.heat_last_error())
            got.append(s.state() / f)
    assert np.linalg.norm(got[0] - got[1]) <= 2 * bar * np.linalg.norm(got[0])
