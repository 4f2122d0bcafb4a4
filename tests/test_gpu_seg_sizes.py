"""A segment size is taken as it is under every variant but the default forms: 512
and 513 nodes are the same whole levels of 16 x 4, 32 x 4 and 16 x 2 tiles, so the same
tiles and the same fields, bit for bit."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,variant", [("fp32_refined", 15), ("fp32_refined", 1), ("fp32_refined", 4),
                                               ("fp32_refined", 9), ("fp64", 2)])
def test_512_nodes_are_512_nodes(precision, variant):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(37, 31, 40, seed=21, dirichlet={2: 0.5}, flux={5: 1.0}, theta=0.5, dt=0.01, nsteps=1, rtol=1e-10,
                     contrast=(0.1, 10.0))
    old, got = hg.heat_tuning_get(), {}
    try:
        for seg in (512, 513):
            t = hg.heat_tuning_get()
            t["variant"][hg.PRECISIONS[precision]], t["seg_nodes"] = variant, [seg] * 3
            hg.heat_tuning_set(t["variant"], t["seg_nodes"], t["pw_quads"])
            with hg.Simulation.from_problem(p, precision=precision) as s:
                assert s.step(1)["status"] == 0
                got[seg] = s.state()
    finally:
        hg.heat_tuning_set(old["variant"], old["seg_nodes"], old["pw_quads"], old["open_w"], old["loop"])
    assert np.array_equal(got[512], got[513])
