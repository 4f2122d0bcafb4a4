"""k_update with several work items per block (loaded a block ahead of the
item's sum, counted once) against one item per block, on a mesh that streams
and whose node count is no multiple of 4. Either solution is within the
precision's bar (1e-9, 1e-8) of the exact one, so they differ by at most twice
that."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision,pid,variant,bar", [("fp64", 0, -1, 1e-9), ("fp32_refined", 1, 15, 1e-8)])
def test_many_items_per_block_equal_one(precision, pid, variant, bar):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(96, 88, 86, seed=9, dirichlet={4: 0.5}, flux={5: 1.0}, theta=0.5, dt=0.002, nsteps=1, rtol=1e-11,
                     contrast=(0.1, 10.0))
    old, got = hg.heat_tuning_get(), {}
    try:
        for quads in (1, 4):  # 734 items of 1024 nodes on 456 or 608 blocks; 184 items of 4096
            t = hg.heat_tuning_get()
            t["variant"][pid], t["pw_quads"][pid] = variant, quads
            hg.heat_tuning_set(t["variant"], t["seg_nodes"], t["pw_quads"])
            with hg.Simulation.from_problem(p, precision=precision) as s:
                assert s.step(1)["status"] == 0
                got[quads] = s.state()
    finally:
        hg.heat_tuning_set(old["variant"], old["seg_nodes"], old["pw_quads"], old["open_w"], old["loop"])
    assert np.linalg.norm(got[1] - got[4]) <= 2 * bar * np.linalg.norm(got[4])
