"""Device arrays that kernels cannot take where they lie: a C caller's array on a
4-byte boundary is taken by a copy, for coefficients, a state in and a state out,
with the results of the same values on an 8-byte boundary, bit for bit."""
import ctypes as C

import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _at(values, offset):
    """A device copy of `values` that starts `offset` bytes into its buffer: (buffer, address)."""
    raw = np.ascontiguousarray(values, dtype=np.float64).view(np.uint8)
    buf = torch.zeros(raw.size + 16, dtype=torch.uint8, device="cuda")
    buf[offset:offset + raw.size] = torch.tensor(raw)
    return buf, C.c_void_p(buf.data_ptr() + offset)


@pytest.mark.parametrize("precision", ["fp64", "fp32_refined"])
@pytest.mark.parametrize("dims", [(1, 1, 1), (9, 7, 11)])
def test_an_array_off_the_8_byte_boundary(dims, precision):
    import paper_1905_07622_gb300 as hg
    from paper_1905_07622_gb300 import api
    p = W.random_box(*dims, seed=2, dirichlet={1: 0.25}, flux={3: 1.0}, dt=0.01, nsteps=1, rtol=1e-10)
    rng = np.random.default_rng(3)
    rc, k = rng.uniform(0.1, 10.0, p.n_elems), rng.uniform(0.1, 10.0, p.n_elems)
    u0 = rng.uniform(-1.0, 1.0, p.n_nodes)
    got = []
    for offset in (0, 4):
        bufs, (a, b, u) = zip(*[_at(v, offset) for v in (rc, k, u0)])
        out, at = _at(np.zeros(p.n_nodes), offset)
        torch.cuda.synchronize()
        with hg.Simulation.from_problem(p, precision=precision) as s:
            api._check(api._lib.heat_set_coeffs(s.sim, a, b, 1))
            assert all(np.array_equal(x, y) for x, y in zip(hg.heat_get_coeffs(s.sim, p.n_elems), (rc, k)))
            api._check(api._lib.heat_set_state(s.sim, u, 1))
            assert s.step(1)["status"] == 0
            api._check(api._lib.heat_get_state(s.sim, at, 1))
            seen = out.cpu().numpy()[offset:offset + 8 * p.n_nodes].copy().view(np.float64)
            assert np.array_equal(seen, s.state())
            got.append(seen)
    assert np.array_equal(*got)
