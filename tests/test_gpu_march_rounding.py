"""How far the FP64 operator entry points are from the exact product, formed here
in extended precision: no further than the plain factorised form (the element
coefficients as sums of two rounded products) on the same input, whose error is
1.242e-15 for the right-hand side's scales and 1.196e-15 for the operator's, both
emulated operation by operation, and 2% for the order of the last additions."""
import numpy as np
import pytest

import workloads as W

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _exact(n, h, rc, k, x, sa, sb):
    L = np.longdouble
    h = [L(v) for v in h]
    m1 = [[v / 3, v / 6] for v in h]
    k1 = [[1 / v, -1 / v] for v in h]
    y = np.zeros_like(x, dtype=L)
    X = x.astype(L)
    at = [tuple(slice((c >> d) & 1, ((c >> d) & 1) + n[d]) for d in (2, 1, 0)) for c in range(8)]
    for a in range(8):
        for b in range(8):
            d = [((a ^ b) >> i) & 1 for i in range(3)]
            m = m1[0][d[0]] * m1[1][d[1]] * m1[2][d[2]]
            s = (k1[0][d[0]] * m1[1][d[1]] * m1[2][d[2]] + m1[0][d[0]] * k1[1][d[1]] * m1[2][d[2]]
                 + m1[0][d[0]] * m1[1][d[1]] * k1[2][d[2]])
            y[at[a]] += (L(sa) * m * rc + L(sb) * s * k) * X[at[b]]
    return y


@pytest.mark.parametrize("sb,plain", [(-0.5, 1.242e-15), (0.5, 1.196e-15)])
def test_error_is_that_of_the_plain_form(sb, plain):
    import paper_1905_07622_gb300 as hg
    n, h = (40, 40, 40), (1 / 100,) * 3
    p = W.random_box(*n, seed=0, extent=(0.4, 0.4, 0.4))
    inside = np.random.default_rng(0).random((40, 40, 40)) < 0.05
    rc, k = np.where(inside, 3.0, 1.0), np.where(inside, 10.0, 1.0)
    z, y, x = np.meshgrid(*[np.linspace(0, 1, 41)] * 3, indexing="ij")
    v = np.cos(3 * x) * np.cos(2 * y + 0.3) * np.cos(5 * z) + 0.5
    ref = _exact(n, [0.4 / 40] * 3, rc, k, v, 1000.0, sb)
    with hg.Simulation.from_problem(p) as s:
        hg.heat_set_coeffs(s.sim, rc.ravel(), k.ravel(), p.n_elems)
        d = torch.tensor(v.ravel(), device="cuda")
        out = torch.empty_like(d)
        hg.heat_apply_general(s.sim, 1000.0, sb, d, out)
        got = out.cpu().numpy().reshape(v.shape)
    err = float(np.linalg.norm((got - ref).astype(np.float64).ravel()) / np.linalg.norm(ref.astype(np.float64).ravel()))
    assert err <= 1.02 * plain, err
