"""One engine with members held on the chip and members that stream.

A member's results are bitwise its own run's; the autotuner and the iteration
profile, which keep every member iterating, work on such a batch; the profile
rates the streaming launches it times by the bytes of the members they carry."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _boxes(dims, element="q1", nsteps=2):
    ps = [W.random_box(*d, seed=7 + i, dirichlet={4: 0.5}, flux={5: 1.0}, theta=0.5, dt=0.002, nsteps=nsteps,
                       rtol=1e-10, contrast=(0.1, 10.0)) for i, d in enumerate(dims)]
    for p in ps:
        p.element = element
    return ps


class _Batch:
    def __init__(self, ps, precision):
        import paper_1905_07622_gb300 as hg
        self.hg, self.sims = hg, [hg.Simulation.from_problem(p, precision=precision) for p in ps]
        self.b = hg.heat_batch_create([s.sim for s in self.sims])

    def __enter__(self):
        return self

    def __exit__(self, *a):
        self.hg.heat_destroy_batch(self.b)
        for s in self.sims:
            s.close()

    def step(self, n):
        rc, stats = self.hg.heat_batch_step(self.b, n, len(self.sims))
        assert rc == 0, self.hg.heat_last_error()
        return stats


# the last of each streams: more than the chip holds in FP32 (1.1 million nodes) and in FP64 (0.13 million);
# 150 nodes a row is a whole number of 32-lane segments
MIXED = [("fp32_refined", "q1", ((20, 18, 22), (149, 90, 92))), ("fp32_refined", "p1", ((20, 18, 22), (149, 90, 92))),
         ("fp64", "q1", ((14, 12, 16), (64, 60, 62)))]


@pytest.mark.parametrize("precision,element,dims", MIXED)
def test_members_are_bitwise_alone(precision, element, dims):
    import paper_1905_07622_gb300 as hg
    ps = _boxes(dims, element)
    alone = []
    for p in ps:
        with hg.Simulation.from_problem(p, precision=precision) as s:
            assert s.step(p.nsteps)["status"] == 0
            alone.append(s.state())
    with _Batch(ps, precision) as b:
        b.step(2)
        for s, a in zip(b.sims, alone):
            assert np.array_equal(s.state(), a)


def test_tetrahedra_in_32_lane_segments_solve_the_system():
    """The streamed step of tetrahedra on a width of whole 32-lane segments
    against an FP64 step of the same: 1e-8 and 1e-9 from the exact one."""
    import paper_1905_07622_gb300 as hg
    p = _boxes(((149, 90, 92),), "p1", nsteps=1)[0]
    got = {}
    for precision in ("fp64", "fp32_refined"):
        with hg.Simulation.from_problem(p, precision=precision) as s:
            assert s.step(1)["status"] == 0
            got[precision] = s.state()
    a, b = got["fp32_refined"], got["fp64"]
    assert np.linalg.norm(a - b) <= (1e-8 + 1e-9) * np.linalg.norm(b)


@pytest.mark.parametrize("precision,element,dims", [MIXED[0], MIXED[2]])
def test_autotune_and_profile_of_a_mixed_batch(precision, element, dims):
    import paper_1905_07622_gb300 as hg
    old = hg.heat_tuning_get()
    try:
        with _Batch(_boxes(dims, element), precision) as b:
            b.step(1)
            both = hg.heat_batch_profile_iteration(b.b, 50)
            table, ms = hg.heat_batch_autotune(b.b, 8)
            assert ms > 0.0 and table == hg.heat_tuning_get()
        hg.heat_tuning_set(old["variant"], old["seg_nodes"], old["pw_quads"], old["open_w"], old["loop"])
        with _Batch(_boxes(dims[1:], element), precision) as b:
            b.step(1)
            streaming = hg.heat_batch_profile_iteration(b.b, 50)
        for k in ("bytes_apply", "bytes_update"):
            assert both[k] == streaming[k] > 0.0
        assert both["ms_apply"] > 0.0 and both["ms_update"] > 0.0
    finally:
        hg.heat_tuning_set(old["variant"], old["seg_nodes"], old["pw_quads"], old["open_w"], old["loop"])
