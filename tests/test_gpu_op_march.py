"""The operator entry points on meshes that end inside a segment tile.

heat_apply, heat_apply_f32, heat_apply_general and heat_rhs run a warp-segment
march of 30-column tiles with four rows per lane, or one on small meshes.
Checked against the oracle's assembled operator at the bars of the operator
tests (1e-12 relative in FP64, 2e-6 in FP32): meshes one column short of, equal
to and beyond a segment, row counts around 4, one to many levels, and both
elements, with and without fixed faces.
"""
import numpy as np
import pytest

import workloads as W
from oracle import transient

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _rel(got, ref):
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("element", ["q1", "p1"])
@pytest.mark.parametrize("dims,dirichlet", [
    ((1, 1, 1), {}), ((28, 3, 2), {1: 0.5}), ((29, 4, 5), {}), ((30, 5, 1), {4: 1.0, 2: -0.5}),
    ((59, 8, 40), {0: 0.25}), ((61, 31, 33), {5: 1.0}), ((7, 70, 3), {}), ((3, 2, 90), {3: 1.0}),
])
def test_products_and_right_hand_side(dims, dirichlet, element):
    import paper_1905_07622_gb300 as hg
    p = W.random_box(*dims, seed=sum(dims), dirichlet=dirichlet, flux={2: 1.0}, theta=0.5, dt=0.01, nsteps=1,
                     contrast=(0.1, 10.0), extent=(1.0, 0.8, 1.3))
    p.element = element
    S = transient.build_system(p)
    x = np.random.default_rng(7).standard_normal(p.n_nodes)
    free = np.ones(p.n_nodes, dtype=bool)
    g = W.apply_dirichlet_values(p, np.full(p.n_nodes, np.nan))
    free[~np.isnan(g)] = False
    A = S.M / p.dt + p.theta * S.K
    L = S.M / p.dt - (1 - p.theta) * S.K
    ref = np.where(free, A @ np.where(free, x, 0.0), x)
    with hg.Simulation.from_problem(p) as s:
        d = torch.tensor(x, device="cuda")
        y = torch.empty_like(d)
        hg.heat_apply(s.sim, d, y)
        assert _rel(y.cpu().numpy(), ref) <= 1e-12
        y32 = torch.empty_like(d, dtype=torch.float32)
        hg.heat_apply_f32(s.sim, d.float(), y32)
        assert _rel(y32.double().cpu().numpy(), ref) <= 2e-6
        hg.heat_apply_general(s.sim, 0.7, 1.9, d, y)
        assert _rel(y.cpu().numpy(), 0.7 * (S.M @ x) + 1.9 * (S.K @ x)) <= 1e-12
        f = torch.empty_like(d)
        hg.heat_flux_vector(s.sim, f)
        hg.heat_rhs(s.sim, 1, d, y)
        lift = A @ np.where(free, 0.0, np.nan_to_num(g))
        b = np.where(free, L @ x + f.cpu().numpy() - lift, np.nan_to_num(g))
        assert _rel(y.cpu().numpy(), b) <= 1e-12
