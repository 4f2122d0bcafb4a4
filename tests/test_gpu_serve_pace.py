"""A request with long inner solves (a stiff material, an inner tolerance of
1e-12) leaves the chip every 48 iterations, so that phases are read and others
admitted: two launches for each. The result stays bitwise the one of the
simulation alone, whose solves are whole."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("element", ["q1", "p1"])
def test_long_inner_solves_let_the_server_look(element):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(18, 17, 20, seed=3, dirichlet={4: 0.5}, flux={5: 1.0}, theta=1.0, dt=10.0, nsteps=4, rtol=1e-10)
    p.k = 10.0 ** np.random.default_rng(1).uniform(-3.0, 3.0, p.n_elems)
    p.element = element
    kw = dict(precision="fp32_refined", inner_rtol=1e-12)
    with hg.Simulation.from_problem(p, **kw) as s:
        assert s.step(p.nsteps)["status"] == 0
        alone = s.state()
    srv = hg.heat_server_create(1 << 30, 4)
    try:
        req, keep = hg.make_request(p, **kw)
        u, st, _ = hg.heat_wait(srv, hg.heat_submit(srv, req), p.n_nodes, timeout_s=60.0)
        launches = hg.heat_server_get_stats(srv)["kernel_launches"]
    finally:
        hg.heat_destroy_server(srv)
    assert np.array_equal(u, alone)
    assert st["iters"] >= 20 * 48  # else no solve was long
    assert launches >= 2 * st["iters"] / 48, (launches, st["iters"])
