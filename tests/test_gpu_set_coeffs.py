"""Coefficients from device arrays, read where they lie (here on an odd 8-byte
boundary), and from host arrays, staged: the same stored values and the same
step, bit for bit; a bad device entry leaves both as they were."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (5, 3, 7), (33, 21, 17)])
def test_device_and_host_coefficients_agree(dims, precision):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(*dims, seed=3, dirichlet={4: 0.5}, flux={5: 1.0}, dt=0.01, nsteps=1, rtol=1e-10)
    rng = np.random.default_rng(5)
    ne = dims[0] * dims[1] * dims[2]
    rc, k = rng.uniform(0.1, 10.0, ne), rng.uniform(0.1, 10.0, ne)
    out = []
    for device in (False, True):
        with hg.Simulation.from_problem(p, precision=precision) as s:
            if device:
                buf = torch.zeros(2 * ne + 3, dtype=torch.float64, device="cuda")
                buf[1:ne + 1], buf[ne + 2:2 * ne + 2] = torch.tensor(rc), torch.tensor(k)
                hg.heat_set_coeffs(s.sim, buf[1:ne + 1], buf[ne + 2:2 * ne + 2], ne)
                bad = torch.ones(ne, dtype=torch.float64, device="cuda")
                bad[ne // 2] = float("nan")
                with pytest.raises(hg.HeatError):
                    hg.heat_set_coeffs(s.sim, bad, bad, ne)
            else:
                hg.heat_set_coeffs(s.sim, rc, k, ne)
            got = hg.heat_get_coeffs(s.sim, ne)
            assert np.array_equal(np.asarray(got[0]), rc) and np.array_equal(np.asarray(got[1]), k)
            s.step(1)
            out.append(s.state())
    assert np.array_equal(out[0], out[1])
