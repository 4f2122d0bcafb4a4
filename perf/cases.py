"""The work whose speed is measured: a user's calls through the public entry points.

Six kinds of work:

  apply     one operator product y = A' x on device vectors (heat_apply, heat_apply_f32): a caller's own
            Krylov or adjoint loop around the operator
  rhs       one right-hand side of the step system (heat_rhs)
  steps     implicit time steps of one simulation from a given field (heat_set_state, heat_step,
            heat_get_state), FP64 or FP32 with refinement, trilinear boxes or six tetrahedra per box;
            with "new" the per-element coefficients are set first (heat_set_coeffs): a new material
  batch     independent samples of one material law advanced together (heat_batch_step)
  plates    the forward models of one proposal per chain of the corrosion inverse problem: each member's
            coefficients from its depth (heat_set_coeffs_corrosion), then the heating period in one batch
  serve     a burst of requests of mixed sizes through the request server, host arrays in and out

Every input comes from the seed alone. `exact` solves the same systems in 64 bits with plain torch.
"""
import math

import numpy as np
import torch

import paper_1905_07622_gb300 as hg

FP64, REFINED = "fp64", "fp32_refined"


# ------------------------------------------------------------------ the cases

def _case(name, kind, nx, ny, nz, field="lognormal", bc="flux", precision=REFINED, element="q1", steps=1, theta=0.5,
          dt=1e-3, members=1, new=False, stretch=False):
    c = {"kind": kind, "nx": nx, "ny": ny, "nz": nz, "field": field, "bc": bc, "precision": precision,
         "element": element, "steps": steps, "theta": theta, "dt": dt, "members": members, "new": new,
         "stretch": stretch}
    return dict(c, name=name) if name else c


def listed():
    return [
        # a caller's own loop on a small ragged mesh: the launch is most of it
        _case("apply_small_ragged", "apply", 33, 21, 17, bc="fixed", precision=FP64, stretch=True),
        # the FP32 operator on the largest configured mesh: memory-bound
        _case("apply_f32_200", "apply", 200, 200, 200, field="layered", bc="bottom", dt=5e-4),
        # the right-hand side on the mesh of the paper's scale (1.03 million unknowns)
        _case("rhs_100", "rhs", 100, 100, 100, field="inclusions", precision=FP64),
        # the smallest configured workload, whole: 20 backward-Euler steps, latency-bound
        _case("steps_two_phase_16", "steps", 16, 16, 16, field="two_phase", bc="side", precision=FP64, steps=20,
              theta=1.0),
        # the headline workload's mesh, material and options, its first steps
        _case("steps_inclusions_100", "steps", 100, 100, 100, field="inclusions", steps=4),
        # the same in FP64 throughout: the parity path
        _case("steps_inclusions_100_f64", "steps", 100, 100, 100, field="inclusions", precision=FP64, steps=1),
        # the stiffest and largest configured workload: a 1:1000 laminate with 8.1 million unknowns
        _case("steps_layered_200", "steps", 200, 200, 200, field="layered", bc="bottom", steps=1, dt=5e-4),
        # the paper's own element on a box that is ragged in every direction
        _case("steps_tetrahedra_ragged", "steps", 77, 50, 61, field="two_phase", element="p1", steps=3, stretch=True),
        # Monte Carlo over a random material: 64 samples of 40^3 in one batch
        _case("batch_lognormal_64x40", "batch", 40, 40, 40, members=64, steps=2, dt=2e-3),
        # one proposal per chain of the inverse problem on its plate
        _case("plates_8", "plates", 64, 20, 64, bc="laser", members=8, steps=5, dt=0.1),
        # a new material on a kept mesh: coefficients in, two steps, field out
        _case("new_material_80", "steps", 80, 80, 80, steps=2, new=True),
        # a burst of mid-size requests to the server
        _case("serve_burst_8", "serve", 48, 48, 48, field="two_phase", members=8, steps=12),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["apply", "apply", "rhs", "steps", "steps", "steps", "batch", "plates", "serve"])
    field = rng.choice(["two_phase", "inclusions", "lognormal", "layered"])
    bc = rng.choice(["flux", "side", "bottom", "fixed"])
    stretch = rng.random() < 0.5
    if kind in ("apply", "rhs"):
        n = [_log_int(rng, 8, 200) for _ in range(3)]
        prec = FP64 if kind == "rhs" else rng.choice([FP64, REFINED])
        return _case(None, kind, *n, field=field, bc=bc, precision=prec, theta=rng.choice([0.5, 1.0]), stretch=stretch,
                     element=rng.choice(["q1", "q1", "q1", "p1"]))
    if kind == "steps":
        prec = rng.choice([FP64, REFINED, REFINED])
        hi = 110 if prec == REFINED else 80
        # a cube of edge n, ragged by up to a fifth in each direction
        n = _log_int(rng, 12, hi)
        d = [max(8, int(n * rng.uniform(0.8, 1.2))) for _ in range(3)]
        return _case(None, "steps", *d, field=rng.choice(["two_phase", "inclusions", "lognormal"]), bc=bc,
                     precision=prec, element=rng.choice(["q1", "q1", "p1"]), steps=rng.randint(1, 4),
                     theta=rng.choice([0.5, 1.0]), dt=rng.choice([5e-4, 1e-3, 2e-3]), new=rng.random() < 0.4,
                     stretch=stretch)
    if kind == "batch":
        n = rng.randint(16, 44)
        return _case(None, "batch", n, n, n, field=rng.choice(["two_phase", "lognormal"]), members=_log_int(rng, 4, 64),
                     steps=rng.randint(1, 3), dt=2e-3)
    if kind == "plates":
        s = rng.uniform(0.5, 1.0)
        return _case(None, "plates", int(64 * s), int(20 * s), int(64 * s), bc="laser", members=rng.randint(2, 12),
                     steps=rng.randint(2, 6), dt=0.1)
    n = rng.randint(20, 56)
    return _case(None, "serve", n, n, n, field="two_phase", members=rng.randint(2, 8), steps=rng.randint(4, 14))


# ------------------------------------------------------------------ inputs

PLATE = (40.0, 12.7, 40.0)  # mm
STEEL = {"z0": 20.0, "half_width": 15.0, "rho_c_sound": 3.6e-3, "k_sound": 0.045, "rho_c_corr": 3.5e-3, "k_corr": 0.005}


def _extent(c):
    if c["kind"] == "plates":
        return PLATE
    return (1.0, 0.8, 1.3) if c["stretch"] else (1.0, 1.0, 1.0)


def _sizes(c, m):
    """The mesh of member m: a server's requests differ in size."""
    if c["kind"] != "serve":
        return c["nx"], c["ny"], c["nz"]
    n = max(8, int(round(c["nx"] * (0.6 + 0.8 * m / max(1, c["members"] - 1)))))
    return n, n, n


def _nsteps(c, m):
    return c["steps"] + (m % 3 if c["kind"] == "serve" else 0)


def _boundary(c):
    """(Dirichlet values by face, fluxes by face, steps with flux on)."""
    if c["bc"] == "side":
        return {0: 0.0}, {}, -1
    if c["bc"] == "bottom":
        return {4: 1.0}, {}, -1
    if c["bc"] == "fixed":
        return {1: 0.25, 4: 1.0}, {3: 0.5}, -1
    if c["bc"] == "laser":
        return {}, {}, -1
    return {}, {5: 1.0}, 50


def _generator(seed, m):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 1009 + m)
    return g


def _centroids(n, ext):
    ax = [(torch.arange(k, device="cuda", dtype=torch.float64) + 0.5) / k for k in n]
    return ax[0][None, None, :], ax[1][None, :, None], ax[2][:, None, None]


def _material(c, n, seed, m):
    """(rho_c, k) of member m, one value per element (flat, x fastest)."""
    g = _generator(seed, m)
    nx, ny, nz = n
    shape = (nz, ny, nx)
    one = torch.ones(shape, dtype=torch.float64, device="cuda")
    if c["field"] == "lognormal":
        k = torch.exp(torch.randn(shape, generator=g, dtype=torch.float64, device="cuda"))
        return one.reshape(-1), k.reshape(-1)
    if c["field"] == "two_phase":
        b = torch.rand(shape, generator=g, dtype=torch.float64, device="cuda") < 0.3
        return torch.where(b, 2.0 * one, one).reshape(-1), torch.where(b, 10.0 * one, one).reshape(-1)
    cx, cy, cz = _centroids(n, None)
    if c["field"] == "inclusions":
        inside = torch.zeros(shape, dtype=torch.bool, device="cuda")
        r = torch.rand((200, 4), generator=g, dtype=torch.float64, device="cuda").cpu().tolist()
        for x, y, z, s in r:
            inside |= (cx - x) ** 2 + (cy - y) ** 2 + (cz - z) ** 2 <= (0.02 + 0.04 * s) ** 2
        return torch.where(inside, 3.0 * one, one).reshape(-1), torch.where(inside, 10.0 * one, one).reshape(-1)
    # layers with conductivity 1 and 1000 in turn, ellipsoidal pockets of an insulator
    layers = max(2, nz // 10)
    cuts = 1 + torch.randperm(nz - 1, generator=g, device="cuda")[: layers - 1].sort().values
    layer = torch.searchsorted(cuts, torch.arange(nz, device="cuda"), right=True)
    k = torch.where(layer % 2 == 0, 1.0, 1000.0).double()[:, None, None].expand(shape).clone()
    rho = one.clone()
    r = torch.rand((30, 6), generator=g, dtype=torch.float64, device="cuda").cpu().tolist()
    pocket = torch.zeros(shape, dtype=torch.bool, device="cuda")
    for x, y, z, a, b, d in r:
        a, b, d = 0.02 + 0.08 * a, 0.02 + 0.08 * b, 0.02 + 0.08 * d
        pocket |= ((cx - x) / a) ** 2 + ((cy - y) / b) ** 2 + ((cz - z) / d) ** 2 <= 1.0
    k[pocket] = 0.01
    rho[pocket] = 0.5
    return rho.reshape(-1), k.reshape(-1)


def _field(c, n, seed, m):
    """The initial temperature of member m: ambient plus a few smooth modes (node order, x fastest)."""
    nx, ny, nz = n
    if c["kind"] == "plates":
        return torch.zeros((nx + 1) * (ny + 1) * (nz + 1), dtype=torch.float64, device="cuda")
    g = _generator(seed, 5000 + m)
    a = torch.rand((4, 7), generator=g, dtype=torch.float64, device="cuda").cpu().tolist()
    ax = [torch.arange(k + 1, device="cuda", dtype=torch.float64) / k for k in n]
    u = torch.zeros((nz + 1, ny + 1, nx + 1), dtype=torch.float64, device="cuda")
    for r in a:
        w = [torch.cos(math.pi * (1 + int(3 * r[d])) * (ax[d] + r[3 + d])) for d in range(3)]
        u += r[6] * w[0][None, None, :] * w[1][None, :, None] * w[2][:, None, None]
    return (u + 0.5).reshape(-1)


def _vector(c, n, seed):
    """What a Krylov loop multiplies: a rough vector without structure."""
    nn = (n[0] + 1) * (n[1] + 1) * (n[2] + 1)
    return torch.randn(nn, generator=_generator(seed, 9000), dtype=torch.float64, device="cuda")


def _depths(c, seed):
    r = np.random.default_rng(int(seed))
    return [float(x) for x in r.uniform(0.0, PLATE[1], c["members"])]


def _laser(c):
    """Flux densities of the front face (y = 0), x fastest: a 10 W spot of 2 mm."""
    nx, nz = c["nx"], c["nz"]
    x = (np.arange(nx) + 0.5) * PLATE[0] / nx
    z = (np.arange(nz) + 0.5) * PLATE[2] / nz
    X, Z = np.meshgrid(x, z)
    return (10.0 / (2.0 * np.pi * 4.0) * np.exp(-((X - 20.0) ** 2 + (Z - 20.0) ** 2) / 8.0)).ravel()


# ------------------------------------------------------------------ the program's side

class _Work:
    """What a program keeps between calls; its handles are given back with it."""

    def __init__(self, case):
        self.case, self.sims, self.meshes, self.batch, self.server = case, [], [], None, None

    def __del__(self):
        hg.heat_destroy_batch(self.batch)
        hg.heat_destroy_server(self.server)
        for s in self.sims:
            hg.heat_destroy_sim(s)
        for m in self.meshes:
            hg.heat_destroy_mesh(m)


class _Request:
    """One request of a client, as hg.make_request takes it."""

    def __init__(self, c, n, rho_c, k, u0, steps):
        self.nx, self.ny, self.nz = n
        self.origin, self.extent = (0.0, 0.0, 0.0), _extent(c)
        self.rho_c, self.k, self.u0 = rho_c.cpu().numpy(), k.cpu().numpy(), u0.cpu().numpy()
        self.dirichlet, self.flux, self.flux_steps = _boundary(c)
        self.theta, self.dt, self.rtol, self.nsteps, self.element = c["theta"], c["dt"], 1e-10, steps, c["element"]


def prepare(case, seed):
    w = _Work(case)
    if case["kind"] == "serve":
        w.server = hg.heat_server_create(16 << 30, 64)
        w.requests = []
        for m in range(case["members"]):
            n = _sizes(case, m)
            rho_c, k = _material(case, n, seed, m)
            w.requests.append((hg.make_request(_Request(case, n, rho_c, k, _field(case, n, seed, m), _nsteps(case, m)),
                                               precision=case["precision"]), (n[0] + 1) * (n[1] + 1) * (n[2] + 1)))
        return w
    dirichlet, flux, flux_steps = _boundary(case)
    params = hg.heat_params_default(theta=case["theta"], dt=case["dt"], rtol=1e-10, precision=case["precision"],
                                    element=case["element"])
    n = _sizes(case, 0)
    w.nn, w.ne = (n[0] + 1) * (n[1] + 1) * (n[2] + 1), n[0] * n[1] * n[2]
    w.material, w.u0, w.out = [], [], []
    for m in range(case["members"]):
        w.meshes.append(hg.heat_create_mesh(*n, (0.0, 0.0, 0.0), _extent(case)))
        w.sims.append(hg.heat_sim_create(w.meshes[-1], hg.make_bc(dirichlet, flux, flux_steps), params))
        if case["kind"] == "plates":
            hg.heat_set_face_flux(w.sims[-1], 2, _laser(case))
        else:
            rho_c, k = _material(case, n, seed, m)
            hg.heat_set_coeffs(w.sims[-1], rho_c, k, w.ne)
            w.material.append((rho_c, k) if case["new"] else None)
        if case["kind"] not in ("apply", "rhs"):
            w.u0.append(_field(case, n, seed, m))
            w.out.append(torch.empty_like(w.u0[-1]))
    if case["kind"] == "plates":
        w.geometry, w.depths = hg.make_corrosion(**STEEL), _depths(case, seed)
    if case["kind"] in ("batch", "plates"):
        w.batch = hg.heat_batch_create(w.sims)
    if case["kind"] == "apply":
        w.x = _vector(case, n, seed)
        if case["precision"] != FP64:
            w.x = w.x.float()
        w.out.append(torch.empty_like(w.x))
    if case["kind"] == "rhs":
        w.u0.append(_field(case, n, seed, 0))
        w.out.append(torch.empty_like(w.u0[0]))
    return w


def run(w):
    c = w.case
    if c["kind"] == "apply":
        (hg.heat_apply if c["precision"] == FP64 else hg.heat_apply_f32)(w.sims[0], w.x, w.out[0])
        return w.out[0]
    if c["kind"] == "rhs":
        hg.heat_rhs(w.sims[0], 1, w.u0[0], w.out[0])
        return w.out[0]
    if c["kind"] == "serve":
        tickets = [hg.heat_submit(w.server, req) for (req, _), _ in w.requests]
        return [hg.heat_wait(w.server, t, nn)[0] for t, (_, nn) in zip(tickets, w.requests)]
    for m, sim in enumerate(w.sims):
        if c["kind"] == "plates":
            hg.heat_set_coeffs_corrosion(sim, w.geometry, w.depths[m])
        elif c["new"]:
            hg.heat_set_coeffs(sim, *w.material[m], w.ne)
        hg.heat_set_state(sim, w.u0[m], w.nn)
    if w.batch is not None:
        status, _ = hg.heat_batch_step(w.batch, c["steps"], len(w.sims))
        if status != hg.HEAT_OK:
            raise hg.HeatError(status, hg.heat_last_error())
    else:
        hg.heat_step(w.sims[0], c["steps"])
    return [hg.heat_get_state(sim, w.nn, out=out) for sim, out in zip(w.sims, w.out)]


def work(case):
    """One operator product reads a vector and the coefficients and writes a vector; a CG iteration of a
    step (about 50 of them, counted once each) cannot do without the product and the update of x, r and d."""
    by = fl = 0.0
    size = 8 if case["precision"] == FP64 else 4
    for m in range(case["members"]):
        n = _sizes(case, m)
        nn, ne = (n[0] + 1) * (n[1] + 1) * (n[2] + 1), n[0] * n[1] * n[2]
        if case["kind"] in ("apply", "rhs"):
            by += 2 * size * nn + 2 * size * ne
            fl += 70.0 * nn
        else:
            its = 700 if case["field"] == "layered" else 50
            by += _nsteps(case, m) * its * (10 * size * nn + 2 * size * ne)
            fl += _nsteps(case, m) * its * 80.0 * nn
    return {"bytes": by, "flops": fl}


# ------------------------------------------------------------------ the same in 64 bits, plain torch

def _box_matrices(h, element):
    """The 8 x 8 mass and stiffness matrices of a box, corner c = x + 2y + 4z."""
    M, K = np.zeros((8, 8)), np.zeros((8, 8))
    if element == "q1":
        m1 = [d / 6.0 * np.array([[2.0, 1.0], [1.0, 2.0]]) for d in h]
        k1 = [1.0 / d * np.array([[1.0, -1.0], [-1.0, 1.0]]) for d in h]
        kron = lambda a, b, d: np.kron(d, np.kron(b, a))  # noqa: E731  (x fastest)
        return kron(*m1), kron(k1[0], m1[1], m1[2]) + kron(m1[0], k1[1], m1[2]) + kron(m1[0], m1[1], k1[2])
    for path in ((1, 2, 4), (1, 4, 2), (2, 1, 4), (2, 4, 1), (4, 1, 2), (4, 2, 1)):
        v = [0, path[0], path[0] + path[1], 7]
        X = np.array([[1.0] + [h[d] * ((c >> d) & 1) for d in range(3)] for c in v])
        vol = abs(np.linalg.det(X)) / 6.0
        grad = np.linalg.inv(X)[1:, :]
        for a in range(4):
            for b in range(4):
                M[v[a], v[b]] += vol * (0.1 if a == b else 0.05)
                K[v[a], v[b]] += vol * grad[:, a] @ grad[:, b]
    return M, K


class _System:
    """(sa M + sb K) on a box mesh and the step system around it."""

    def __init__(self, c, n, rho_c, k):
        self.c, self.n = c, n
        nx, ny, nz = n
        ext = _extent(c)
        self.h = [ext[d] / n[d] for d in range(3)]
        M, K = _box_matrices(self.h, c["element"])
        self.M, self.K = (torch.tensor(a, device="cuda") for a in (M, K))
        self.rho_c, self.k = rho_c.reshape(nz, ny, nx), k.reshape(nz, ny, nx)
        self.shape = (nz + 1, ny + 1, nx + 1)
        self.corners = [(slice(z, z + nz), slice(y, y + ny), slice(x, x + nx))
                        for z in (0, 1) for y in (0, 1) for x in (0, 1)]
        dirichlet, self.flux, self.flux_steps = _boundary(c)
        self.free = torch.ones(self.shape, dtype=torch.bool, device="cuda")
        self.g = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        for f in sorted(dirichlet, reverse=True):  # the lowest face wins
            at = self._face(f)
            self.free[at] = False
            self.g[at] = dirichlet[f]
        self.F = self._loads()

    def _face(self, f):
        at = [slice(None)] * 3
        at[2 - f // 2] = 0 if f % 2 == 0 else -1
        return tuple(at)

    def _loads(self):
        F = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        loads = dict(self.flux)
        if self.c["kind"] == "plates":
            loads[2] = torch.tensor(_laser(self.c), device="cuda").reshape(self.n[2], self.n[0])
        for f, q in loads.items():
            a, b = [d for d in range(3) if d != f // 2]  # a is the faster index of the face
            area = self.h[a] * self.h[b]
            face = torch.zeros((self.n[b] + 1, self.n[a] + 1), dtype=torch.float64, device="cuda")
            for i in (0, 1):
                for j in (0, 1):
                    # trilinear boxes: a quarter to each corner; tetrahedra cut the quad along its lower-upper
                    # diagonal, whose ends belong to both triangles
                    share = 0.25 if self.c["element"] == "q1" else (1.0 / 3.0 if i == j else 1.0 / 6.0)
                    face[j:j + self.n[b], i:i + self.n[a]] += q * area * share
            F[self._face(f)] += face
        return F

    def product(self, sa, sb, x):
        nx, ny, nz = self.n
        xe = torch.stack([x[at].reshape(-1) for at in self.corners])
        ye = sa * self.rho_c.reshape(1, -1) * (self.M @ xe) + sb * self.k.reshape(1, -1) * (self.K @ xe)
        y = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        for c, at in enumerate(self.corners):
            y[at] += ye[c].reshape(nz, ny, nx)
        return y

    def eliminated(self, x):
        y = self.product(1.0 / self.c["dt"], self.c["theta"], torch.where(self.free, x, 0.0))
        return torch.where(self.free, y, x)

    def right_side(self, u, step):
        b = self.product(1.0 / self.c["dt"], self.c["theta"] - 1.0, u)
        if self.flux_steps < 0 or step <= self.flux_steps:
            b = b + self.F
        b = b - self.product(1.0 / self.c["dt"], self.c["theta"], torch.where(self.free, 0.0, self.g))
        return torch.where(self.free, b, self.g)

    def diagonal(self):
        d = torch.zeros(self.shape, dtype=torch.float64, device="cuda")
        for c, at in enumerate(self.corners):
            d[at] += self.rho_c / self.c["dt"] * self.M[c, c] + self.c["theta"] * self.k * self.K[c, c]
        return torch.where(self.free, d, 1.0)

    def solve(self, b, x):
        """Conjugate gradients to rounding, with the residual formed anew now and then."""
        pinv = 1.0 / self.diagonal()
        b0 = torch.where(self.free, b, 0.0)
        x = torch.where(self.free, x, self.g)
        goal = 1e-28 * float((b0 * pinv * b0).sum())
        for _ in range(4):
            r = torch.where(self.free, b - self.eliminated(x), 0.0)
            d = pinv * r
            delta = (r * d).sum()
            for it in range(4000):
                if it % 10 == 0 and float(delta) <= goal:
                    break
                q = torch.where(self.free, self.eliminated(d), 0.0)
                alpha = delta / (d * q).sum()
                x = x + alpha * d
                r = r - alpha * q
                z = pinv * r
                new = (r * z).sum()
                d = z + (new / delta) * d
                delta = new
            if it == 0:
                break
            goal = max(goal, 1e-30 * float((b0 * pinv * b0).sum()))
            if self.c["field"] == "layered":
                break
        return x

    def march(self, u, steps):
        u = torch.where(self.free, u.reshape(self.shape), self.g)
        for s in range(1, steps + 1):
            u = self.solve(self.right_side(u, s), u)
        return u.reshape(-1)


def _corroded(c, n, depth):
    """(rho_c, k) of the plate with a parabolic crevice of this depth from the rear face."""
    nx, ny, nz = n
    zc = (np.arange(nz) + 0.5) * (PLATE[2] / nz)
    t = (zc - STEEL["z0"]) / STEEL["half_width"]
    reach = depth * (1.0 - t * t)
    yc = (np.arange(ny) + 0.5) * (PLATE[1] / ny)
    bad = (np.abs(t) < 1.0)[:, None] & ((PLATE[1] - yc)[None, :] < reach[:, None])
    bad = torch.tensor(bad, device="cuda")[:, :, None].expand(nz, ny, nx)
    full = lambda a, b: torch.where(bad, torch.tensor(a, dtype=torch.float64, device="cuda"),  # noqa: E731
                                    torch.tensor(b, dtype=torch.float64, device="cuda")).reshape(-1)
    return full(STEEL["rho_c_corr"], STEEL["rho_c_sound"]), full(STEEL["k_corr"], STEEL["k_sound"])


def exact(case, seed):
    n = _sizes(case, 0)
    if case["kind"] in ("apply", "rhs"):
        s = _System(case, n, *_material(case, n, seed, 0))
        if case["kind"] == "apply":
            x = _vector(case, n, seed)
            x = x if case["precision"] == FP64 else x.float().double()
            return s.eliminated(x.reshape(s.shape)).reshape(-1)
        return s.right_side(_field(case, n, seed, 0).reshape(s.shape), 1).reshape(-1)
    out = []
    depths = _depths(case, seed) if case["kind"] == "plates" else []
    for m in range(case["members"]):
        if case["kind"] in ("batch", "plates", "serve") and m not in (0, case["members"] - 1):
            out.append(None)  # the first and the last member stand for all
            continue
        n = _sizes(case, m)
        mat = _corroded(case, n, depths[m]) if case["kind"] == "plates" else _material(case, n, seed, m)
        out.append(_System(case, n, *mat).march(_field(case, n, seed, m), _nsteps(case, m)))
    return out
