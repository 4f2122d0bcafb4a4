"""poll_period on meshes held on the chip: a launch ends after that many
iterations (at least the six of a streaming tick) when it is below the default,
and the next takes the iteration up where it stood. Where launches end must not
show in the results: every state and count is bitwise the one of whole inner
solves, for both elements, one box and many, a mesh split in x, a solve that
crosses FP64's true residual, and plain FP32."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(p, precision, poll):
    import paper_1905_07622_gb300 as hg
    with hg.Simulation.from_problem(p, precision=precision, poll_period=poll) as s:
        out, its, launches = [], [], 0
        for _ in range(p.nsteps):
            st = s.step(1)
            assert st["status"] == 0
            out.append(s.state())
            its.append((st["iters"], st["outer"]))
            launches += st["kernel_launches"]
        return out, its, launches


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined", "fp32_plain"])
@pytest.mark.parametrize("element,dims", [("q1", (12, 10, 14)), ("p1", (12, 10, 14)), ("q1", (37, 31, 29)),
                                          ("p1", (33, 30, 31)), ("q1", (150, 6, 7))])
def test_a_solve_cut_into_launches_is_bitwise_the_whole_one(element, dims, precision):
    p = W.random_box(*dims, seed=3, dirichlet={4: 1.0}, flux={3: 0.5}, theta=0.5, dt=0.5, nsteps=2,
                     rtol=1e-6 if precision == "fp32_plain" else 1e-10, contrast=(0.05, 20.0))
    p.element = element
    whole, its, launches = _run(p, precision, 32)
    for poll in (1, 7, 20):
        cut, cut_its, cut_launches = _run(p, precision, poll)
        assert cut_its == its, poll
        for n in range(p.nsteps):
            assert np.array_equal(cut[n], whole[n]), (poll, n)
        # one launch of the solve, one of the passes and one count per poll_period iterations
        assert cut_launches >= 3 * sum(i for i, _ in its) / max(poll, 6), poll
