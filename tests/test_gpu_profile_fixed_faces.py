"""The iteration profile and the autotuner on meshes with fixed faces that are
held on the chip: their seeded residual is zero on the fixed rows, as a solve's
is, so the iteration they time is one of a symmetric positive system and does
not break down (100 and more iterations on every fixed face)."""
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
@pytest.mark.parametrize("element", ["q1", "p1"])
@pytest.mark.parametrize("faces", [(4,), (0, 3), (0, 1, 2, 3, 4, 5)])
def test_profile_and_tune_with_fixed_faces(faces, element, precision):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(14, 12, 16, seed=7, dirichlet={f: 0.5 for f in faces}, theta=0.5, dt=0.002, nsteps=1,
                     rtol=1e-10, contrast=(0.1, 10.0))
    p.element = element
    old = hg.heat_tuning_get()
    try:
        with hg.Simulation.from_problem(p, precision=precision) as s:
            s.step(1)
            assert hg.heat_profile_iteration(s.sim, 120)["ms_apply"] > 0.0
            assert hg.heat_autotune(s.sim, 5)[1] > 0.0
    finally:
        hg.heat_tuning_set(old["variant"], old["seg_nodes"], old["pw_quads"], old["open_w"], old["loop"])
