"""Turning the Chebyshev passes on and off between steps, where that changes the
work lists: with them a mesh takes 16-lane segments and the streaming kernels,
without them 32-lane segments on some widths (nx + 1 just below a multiple of
30) and the chip where it fits. The switched simulation solves each step like a
new one that was made with that preconditioner and given the same history: both
are within the precision's bar of the exact step, so at most twice that apart."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BARS = {"fp64": 1e-9, "fp32_refined": 1e-8}


def _close(a, b, bar):
    assert np.linalg.norm(a - b) <= 2 * bar * np.linalg.norm(b)


@pytest.mark.parametrize("precision,element,dims,degrees", [
    ("fp32_refined", "q1", (29, 29, 29), (0, 3, 0, 2)),
    ("fp32_refined", "q1", (57, 40, 33), (3, 0, 3, 0)),
    ("fp32_refined", "q1", (59, 21, 17), (0, 2, 0)),
    ("fp32_refined", "p1", (57, 20, 24), (2, 0, 2)),
    ("fp32_refined", "p1", (29, 30, 28), (0, 2, 0)),
    ("fp32_refined", "q1", (149, 90, 92), (0, 2, 0)),  # too large for the chip
    ("fp64", "q1", (29, 29, 29), (0, 2, 0)),
    ("fp64", "q1", (59, 50, 52), (2, 0)),
])
def test_switching_changes_the_work_lists(precision, element, dims, degrees):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(*dims, seed=5, dirichlet={4: 0.5}, flux={5: 1.0}, theta=0.5, dt=0.01, nsteps=1, rtol=1e-11,
                     contrast=(0.1, 10.0))
    p.element = element
    kw = dict(theta=p.theta, dt=p.dt, rtol=p.rtol, precision=precision, element=element)
    with hg.Simulation.from_problem(p, precision=precision) as s:
        for m in degrees:
            s.set_params(cheb_degree=m, **kw)
            history = hg.heat_get_history(s.sim, p.n_nodes)
            assert s.step(1)["status"] == 0
            with hg.Simulation.from_problem(p, precision=precision, cheb_degree=m) as fresh:
                hg.heat_set_history(fresh.sim, *history, p.n_nodes)
                assert fresh.step(1)["status"] == 0
                _close(s.state(), fresh.state(), BARS[precision])


def test_switching_one_member_of_a_batch():
    import paper_1905_07622_gb300 as hg
    ps = [W.random_box(*d, seed=6, dirichlet={4: 0.5}, flux={5: 1.0}, theta=0.5, dt=0.01, nsteps=1, rtol=1e-11,
                       contrast=(0.1, 10.0)) for d in ((29, 29, 29), (57, 20, 24), (12, 10, 14))]
    sims = [hg.Simulation.from_problem(p, precision="fp32_refined") for p in ps]
    try:
        b = hg.heat_batch_create([s.sim for s in sims])
        try:
            for degrees in ((0, 0, 0), (2, 0, 3), (0, 3, 0), (2, 2, 2), (0, 0, 0)):
                history = []
                for s, p, m in zip(sims, ps, degrees):
                    s.set_params(cheb_degree=m, theta=p.theta, dt=p.dt, rtol=p.rtol, precision="fp32_refined")
                    history.append(hg.heat_get_history(s.sim, p.n_nodes))
                rc, _ = hg.heat_batch_step(b, 1, len(sims))
                assert rc == 0, hg.heat_last_error()
                for s, p, m, h in zip(sims, ps, degrees, history):
                    with hg.Simulation.from_problem(p, precision="fp32_refined", cheb_degree=m) as fresh:
                        hg.heat_set_history(fresh.sim, *h, p.n_nodes)
                        assert fresh.step(1)["status"] == 0
                        _close(s.state(), fresh.state(), BARS["fp32_refined"])
        finally:
            hg.heat_destroy_batch(b)
    finally:
        for s in sims:
            s.close()
