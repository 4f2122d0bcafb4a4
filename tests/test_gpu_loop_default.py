"""The persistent iteration under the default variant: loop = 1 takes the place
of the on-chip solve and of the streaming launches alike, as on the plain form
of the same shape (variant 15), whose fields and iteration counts it has bit for
bit."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _run(p, variant, loop):
    import paper_1905_07622_gb300 as hg
    old = hg.heat_tuning_get()
    t = hg.heat_tuning_get()
    t["variant"][1], t["seg_nodes"], t["loop"][1] = variant, [256] * 3, loop
    try:
        hg.heat_tuning_set(t["variant"], t["seg_nodes"], t["pw_quads"], t["open_w"], t["loop"])
        with hg.Simulation.from_problem(p, precision="fp32_refined") as s:
            st = s.step(p.nsteps)
            assert st["status"] == 0
            return s.state(), st["iters"], st["kernel_launches"]
    finally:
        hg.heat_tuning_set(old["variant"], old["seg_nodes"], old["pw_quads"], old["open_w"], old["loop"])


@pytest.mark.parametrize("dims", [(37, 11, 19), (149, 90, 92)])  # fits the chip; streams
def test_loop_has_effect_under_the_default_variant(dims):
    p = W.random_box(*dims, seed=21, dirichlet={2: 0.5}, flux={5: 1.0}, theta=0.5, dt=0.01, nsteps=2, rtol=1e-10,
                     contrast=(0.1, 10.0))
    tick, loop, default = _run(p, 15, 0), _run(p, 15, 1), _run(p, 0, 1)
    assert np.array_equal(loop[0], tick[0]) and np.array_equal(default[0], loop[0])
    assert default[1:] == loop[1:] and default[1] == tick[1]
    assert default[2] < tick[2] / 2
