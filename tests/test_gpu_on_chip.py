"""The inner solve held on the chip (k_cg_res, k_cg_res64).

The kernel cuts a mesh into boxes, one per block, and exchanges one-node halos
and partial sums between them. Checked where that can go wrong: meshes of one
box and of many, boxes that end inside a march segment (30 columns), a row
group (4 rows) or a group of 4 nodes, meshes split in x, Dirichlet faces on
every side, both elements, solves long enough to cross FP64's periodic true
residual, and more rounds than one launch's limit. Every step is held to the
paths' bars against the sparse direct solution (1e-9 in FP64, 1e-8 refined).
A wait that can never end must fail the step and leave the GPU usable.
"""
import numpy as np
import pytest

import pins
import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

BARS = {"fp64": 1e-9, "fp32_refined": 1e-8}


def _steps(p, precision, **kw):
    import paper_1905_07622_gb300 as hg
    with hg.Simulation.from_problem(p, precision=precision, **kw) as s:
        out = []
        for _ in range(p.nsteps):
            assert s.step(1)["status"] == 0
            out.append(s.state())
        return out


def _check(p, precision, us):
    ref = pins.oracle_steps(p)
    for n in range(1, p.nsteps + 1):
        err = np.linalg.norm(us[n - 1] - ref.u[n]) / np.linalg.norm(ref.u[n])
        assert err <= BARS[precision], (n, err)


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
@pytest.mark.parametrize("element", ["q1", "p1"])
@pytest.mark.parametrize("dims,dirichlet", [
    ((1, 2, 1), {}),                                    # one box, one group of 4 nodes
    ((29, 4, 3), {1: 0.5}),                             # exactly one segment of columns
    ((30, 3, 4), {0: 0.5}),                             # one column more
    ((59, 7, 2), {3: 1.0}),                             # two segments, whole row groups
    ((150, 4, 5), {1: 0.5, 4: 1.0}),                    # split in x
    ((18, 31, 3), {2: 0.25}),                           # boxes along y
    ((5, 4, 70), {5: 1.0}),                             # boxes along z
    ((26, 22, 25), {f: 0.1 * f for f in range(6)}),     # every face fixed
])
def test_boxes_match_the_direct_solution(dims, dirichlet, element, precision):
    p = W.random_box(*dims, seed=sum(dims), dirichlet=dirichlet, flux={2: 1.0} if not dirichlet else {}, theta=0.5,
                     dt=0.01, nsteps=2, rtol=1e-11, contrast=(0.1, 10.0), extent=(1.0, 0.8, 1.3))
    p.element = element
    _check(p, precision, _steps(p, precision))


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
def test_long_solves_leave_and_reenter_the_chip(precision):
    """FP64 leaves it for the true residual every 50 iterations and goes on
    with the same direction; the iteration counts stay the oracle's."""
    from oracle import transient
    p = W.random_box(14, 12, 16, seed=4, dt=10.0, contrast=(0.01, 100.0), dirichlet={4: 1.0}, flux={3: 0.5}, nsteps=2,
                     rtol=1e-10)
    ref = transient.run(p, solver="pcg", system=transient.build_system(p))
    assert min(ref.iters) > 50  # every step crosses the residual period
    import paper_1905_07622_gb300 as hg
    with hg.Simulation.from_problem(p, precision=precision) as s:
        us, its = [], []
        for _ in range(p.nsteps):
            its.append(s.step(1)["iters"])
            us.append(s.state())
    _check(p, precision, us)
    if precision == "fp64":
        assert all(abs(a - b) <= 2 for a, b in zip(its, ref.iters)), (its, ref.iters)


def test_rounds_limit_saves_and_resumes_the_iteration():
    """heat_profile_iteration runs 40 rounds a launch: the state it leaves and
    takes up again must be an iteration in progress (it fails otherwise)."""
    import paper_1905_07622_gb300 as hg
    p = W.lognormal_cube(3, n=20, nsteps=1)
    with hg.Simulation.from_problem(p, precision="fp32_refined") as s:
        s.step(1)
        t = hg.heat_profile_iteration(s.sim, 100)
        assert t["ms_apply"] > 0.0 and t["ms_update"] == 0.0


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
def test_a_wait_that_runs_out_fails_the_step_and_the_gpu_stays_usable(precision):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(37, 11, 19, seed=21, dirichlet={2: 0.5}, flux={5: 1.0}, theta=0.5, dt=0.01, nsteps=2, rtol=1e-11)
    hg.heat_debug_loop_wait(1, 0.02)
    try:
        with hg.Simulation.from_problem(p, precision=precision) as s:
            rc, st = hg.heat_step_nocheck(s.sim, 1)
            assert rc == hg.HEAT_ERR_TIMEOUT, (rc, hg.heat_last_error())
            hg.heat_debug_loop_wait(0, 0.0)
            hg.heat_set_history(s.sim, p.u0, None, 0, p.n_nodes)
            us = []
            for _ in range(p.nsteps):
                assert s.step(1)["status"] == 0
                us.append(s.state())
    finally:
        hg.heat_debug_loop_wait(0, 0.0)
    _check(p, precision, us)
