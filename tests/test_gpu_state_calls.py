"""A state set from the host or from the device, and read back on either, is the
same field bit for bit: at once (Dirichlet values imposed), and after steps
(whose result lies in another slot); setting it again starts over."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 3, 7), (33, 21, 17)])
def test_state_by_host_and_device(dims, precision):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(*dims, seed=2, dirichlet={1: 0.25, 4: 0.5}, flux={3: 1.0}, dt=0.01, nsteps=3, rtol=1e-10)
    u0 = np.random.default_rng(3).uniform(-1.0, 1.0, p.n_nodes)
    runs = []
    with hg.Simulation.from_problem(p, precision=precision) as s:
        out = torch.empty(p.n_nodes, dtype=torch.float64, device="cuda")
        for device in (False, True):
            hg.heat_set_state(s.sim, torch.tensor(u0, device="cuda") if device else u0, p.n_nodes)
            seen = []
            for _ in range(3):
                host = np.array(hg.heat_get_state(s.sim, p.n_nodes))
                hg.heat_get_state(s.sim, p.n_nodes, out=out)
                assert np.array_equal(out.cpu().numpy(), host)
                seen.append(host)
                assert s.step(1)["status"] == 0
            assert np.array_equal(seen[0], W.apply_dirichlet_values(p, u0.copy()))
            runs.append(seen)
    assert all(np.array_equal(a, b) for a, b in zip(*runs))
