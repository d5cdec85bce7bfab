"""Performance cases: what a user of the library has it do, through ``Solver`` and ``LtsRun``.

A case names a problem (mesh family and size), the scheme's options and what is
done with it:

  load     the pre-processing phase alone: averages in, WENO + predictor of every element out
  advance  load averages, then run local (or global) steps through ``advance_to``
  steps    load averages, then single ``sweep`` calls whose update count the caller looks at
  restart  restore a saved mid-run state, queue sweeps, wait once
  adjoint  ``LtsRun`` forward and backward (gradient of a kinetic energy)

Meshes are kept per problem and size (a user keeps a mesh); the initial data of
every state come from its seed: the two gas states of the Riemann problems and
explosions and the vortex strength vary by some per cent, the centre too.
"""
import functools
import math
import random

import numpy as np
import torch

from paper_1408_3719_gb300 import adjoint as A
from paper_1408_3719_gb300 import aleweno
from paper_1408_3719_gb300 import workloads as W


def listed():
    return [
        # the paper's Sod tube, second order, one global step for all: many tiny launches
        dict(name="tube_p1_gts_2k", problem="tube", size=2000, do="advance", order=1, gts=True, sweeps=50),
        # the Kidder shell (exact-state boundary, Osher flux), advanced sweep by sweep
        dict(name="kidder_p3_osher_2k", problem="kidder", size=2400, do="steps", order=3, flux="osher", sweeps=25),
        # the smallest vortex of the convergence study, fourth order, local steps
        dict(name="vortex_p3_lts_4k", problem="vortex", size=4050, do="advance", order=3, sweeps=50),
        # the paper's first Riemann problem, third order, Osher flux, local steps
        dict(name="riemann_p2_osher_9k", problem="riemann", size=8862, do="advance", order=2, flux="osher", sweeps=50),
        # pre-processing phase of the middle vortex: every element reconstructed and predicted
        dict(name="vortex_p3_load_16k", problem="vortex", size=16200, do="load", order=3),
        # a mesh at rest (Eulerian), second order, local steps
        dict(name="vortex_p1_eulerian_64k", problem="vortex", size=64082, do="advance", order=1, eulerian=True,
             sweeps=50),
        # the paper's explosion on the stand-in for its mesh m1, third order, Osher flux
        dict(name="explosion_p2_osher_44k", problem="m1", size=44097, do="advance", order=2, flux="osher", sweeps=50),
        # a graded-disc explosion in mid-run, fourth order, continued from a saved state
        dict(name="explosion_p3_restart_134k", problem="disc", size=134192, do="restart", order=3, sweeps=100),
        # the same disc with global steps, third order: every element in every step
        dict(name="explosion_p2_gts_134k", problem="disc", size=134192, do="advance", order=2, gts=True, sweeps=4),
        # independent instances advanced together, third order
        dict(name="batch_p2_16", problem="batch", size=130000, do="advance", order=2, sweeps=25, instances=16),
        # gradient of the kinetic energy in a disc after 50 sweeps, third order
        dict(name="adjoint_p2_disc_50k", problem="vortex", size=49928, do="adjoint", order=2, sweeps=50, radius=1.0),
        # gradient of the whole mesh's kinetic energy, fourth order
        dict(name="adjoint_p3_global_16k", problem="vortex", size=16200, do="adjoint", order=3, sweeps=20, radius=0.0),
    ]


def draw(rng: random.Random):
    def logint(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["tube", "kidder", "vortex", "riemann", "m1", "disc", "batch", "adjoint", "load", "saltzman"])
    flux = rng.choice(["rusanov", "osher"])
    if kind == "tube":
        return dict(problem="tube", size=20 * logint(50, 900), do=rng.choice(["advance", "steps"]),
                    order=rng.choice([1, 2]), gts=rng.random() < 0.5, flux=flux, sweeps=rng.randint(15, 50))
    if kind == "kidder":
        return dict(problem="kidder", size=240 * rng.randint(6, 40), do=rng.choice(["advance", "steps"]),
                    order=rng.choice([2, 3]), gts=rng.random() < 0.3, flux=flux, sweeps=rng.randint(10, 40))
    if kind == "vortex":
        n = logint(20, 160)
        return dict(problem="vortex", size=2 * n * n, do=rng.choice(["advance", "steps", "restart"]),
                    order=rng.choice([1, 2, 3]), flux=flux, eulerian=rng.random() < 0.3, sweeps=rng.randint(15, 60))
    if kind == "riemann":
        return dict(problem="riemann", size=42 * logint(60, 500), do="advance", order=rng.choice([1, 2, 3]),
                    gts=rng.random() < 0.3, flux=flux, sweeps=rng.randint(15, 60))
    if kind == "m1":
        return dict(problem="m1", size=logint(8000, 60000), do="advance", order=rng.choice([1, 2]), flux=flux,
                    sweeps=rng.randint(15, 60))
    if kind == "disc":
        if rng.random() < 0.5:
            return dict(problem="disc", size=logint(12000, 120000), do="restart", order=3,
                        sweeps=rng.randint(30, 100))
        return dict(problem="disc", size=logint(12000, 120000), do="advance", order=2, gts=True,
                    sweeps=rng.randint(1, 4))
    if kind == "batch":
        k = rng.randint(2, 16)
        return dict(problem="batch", size=k * rng.randint(2500, 7500), do="advance", order=rng.choice([1, 2]),
                    sweeps=rng.randint(10, 30), instances=k)
    if kind == "adjoint":
        order = rng.choice([1, 2, 3])
        n = logint(24, 158 if order < 3 else 90)
        return dict(problem="vortex", size=2 * n * n, do="adjoint", order=order,
                    sweeps=rng.randint(5, 50 if order < 3 else 20), radius=rng.choice([0.0, 1.0]))
    if kind == "saltzman":  # moving wall, global steps at first
        return dict(problem="saltzman", size=20 * rng.randint(60, 300), do="advance", order=rng.choice([1, 2]),
                    sweeps=rng.randint(10, 40))
    n = logint(24, 90)
    return dict(problem="vortex", size=2 * n * n, do="load", order=rng.choice([1, 2, 3]), eulerian=rng.random() < 0.3)


# ---------------------------------------------------------------------------
# problems
# ---------------------------------------------------------------------------

@functools.lru_cache(maxsize=24)
def _mesh(problem, size, instances):
    """Mesh (a list of them for a batch) of about `size` triangles."""
    if problem == "tube":
        return W.shock_tube_mesh(size // 20, 10, 1.0, 200.0 / size)
    if problem == "saltzman":
        return W.saltzman(size // 20, 10)[0]
    if problem == "kidder":
        return W.kidder(10, size // 20)[0]
    if problem == "vortex":
        return W.vortex_grid_mesh(int(round(math.sqrt(size / 2))))
    if problem == "riemann":
        return W.tube_mesh_periodic_y(size // 42, 21, ly=21.0 * 42 / size, y0=0.0, jitter=0.0)
    if problem == "m1":
        return W.disc_m1_mesh(0.86 * math.sqrt(44097 / size))
    if problem == "disc":
        return W.disc_mesh(0.0022 * math.sqrt(134192 / size))
    per = size / instances
    rng = random.Random(instances)
    out = []
    for k in range(instances):
        n = per * math.exp(rng.uniform(-0.8, 0.5))
        if k % 2:
            out.append(W.disc_mesh(math.sqrt(0.646 / n), seed=k))
        else:
            out.append(W.shock_tube_mesh(max(10, int(n / 20)), 10, 1.0, 10.0 / max(10, int(n / 20)), seed=k))
    return out


def _inputs(case, seed):
    """(mesh, averages, t_end) of a case; a batch has lists of them."""
    rng = random.Random(seed * 7919 + case["size"])
    mesh = _mesh(case["problem"], case["size"], case.get("instances", 1))
    near = lambda v: v * rng.uniform(0.96, 1.04)  # noqa: E731
    left, right = (near(1.0), 0.0, 0.0, near(1.0)), (near(0.125), 0.0, 0.0, near(0.1))
    rule = W._subtriangle_rule(4)
    if case["problem"] == "tube":
        return mesh, W.cell_average(mesh, lambda x, y: W.riemann_state(x, y, left, right, 0.5, 1.4), rule), 0.2
    if case["problem"] == "riemann":
        return mesh, W.cell_average(mesh, lambda x, y: W.riemann_state(x, y, left, right, 0.0, 1.4), rule), 0.2
    if case["problem"] in ("m1", "disc"):
        r = 0.5 * rng.uniform(0.98, 1.02)
        return mesh, W.cell_average(mesh, lambda x, y: W.explosion_state(x, y, left, right, r, 1.4), rule), 0.25
    if case["problem"] == "saltzman":
        q = W.prim_to_cons(near(1.0), 0.0, 0.0, near(2.0 / 3.0 * 1e-4), 5.0 / 3.0)
        return mesh, np.tile(q, (mesh["tri"].shape[0], 1)), 0.6
    if case["problem"] == "kidder":
        t0 = rng.uniform(0.0, 0.02)  # a state on the exact compression
        q = W.cell_average(mesh, lambda x, y: W.prim_to_cons(*W.kidder_prim(x, y, 0.0), 2.0), W._duffy_rule(4))
        return mesh, q * (1.0 + t0 * np.cos(5.0 * W._corner_coords(mesh).mean(1)[:, :1])), 0.18
    if case["problem"] == "vortex":
        eps, cx, cy = 5.0 * rng.uniform(0.9, 1.05), 5.0 + rng.uniform(-0.2, 0.2), 5.0 + rng.uniform(-0.2, 0.2)
        q = W.cell_average(mesh, lambda x, y: W.prim_to_cons(*W.vortex_prim(x, y, 1.4, eps, (cx, cy)), 1.4),
                           W._duffy_rule(4))
        return mesh, q, 1.0
    qs, ts = [], []
    for k, m in enumerate(mesh):
        lo = (1.0 / rng.uniform(2.0, 8.0), 0.0, 0.0, 1.0 / rng.uniform(2.0, 10.0))
        xd = rng.uniform(0.35, 0.55)
        f = W.explosion_state if k % 2 else W.riemann_state
        qs.append(W.cell_average(m, lambda x, y: f(x, y, left, lo, xd, 1.4), rule))
        ts.append(0.25 if k % 2 else 0.2)
    return mesh, np.concatenate(qs), ts


def _outputs(s):
    """Buffers for the whole LTS state."""
    n, d = s.n_tris, torch.float64
    new = lambda *shape, dt=d: torch.empty(shape, dtype=dt, device="cuda")  # noqa: E731
    return dict(Q=new(n, 4), QM=new(n, 4), HM=new(n, 3), t=new(n, dt=torch.int64), dt=new(n, dt=torch.int64),
                X=new(n, 6), count=new(n, dt=torch.int64), qhat=new(n, s.Nst, 4))


def prepare(case, seed):
    mesh, q, t_end = _inputs(case, seed)
    opt = dict(order_M=case["order"], gts=case.get("gts", False), flux=case.get("flux", "rusanov"),
               eulerian=case.get("eulerian", False))
    batch = case["problem"] == "batch"
    if case["problem"] == "kidder":
        opt.update(gamma=2.0)
    if case["problem"] == "saltzman":
        opt.update(gamma=5.0 / 3.0, wall_velocity=(1.0, 0.0), t_switch=0.01, cfl_start=0.1)
    if case["do"] == "restart" and case["problem"] == "disc":
        opt.update(t_switch=0.01, cfl_start=0.5)
    s = aleweno.Solver(t_end=1.0 if batch else t_end, **opt)
    s.load_batch(mesh, t_end) if batch else s.load_mesh(mesh)
    state = dict(do=case["do"], sweeps=case.get("sweeps", 0), solver=s, t_end=s.t_end)
    if case["do"] == "adjoint":
        state["Q0"] = torch.tensor(q, device="cuda", requires_grad=True)
        state["xy0"] = torch.tensor(mesh["xy"], device="cuda", requires_grad=True)
        c = W._corner_coords(mesh)
        mask = A.disc_mask(c.reshape(-1, 6), (5.0, 5.0), case["radius"]) if case["radius"] else np.ones(len(q))
        state["mask"] = torch.tensor(mask, device="cuda")
        return state
    state["out"] = _outputs(s)
    state["Q0"] = torch.tensor(q, device="cuda")
    if case["do"] == "restart":
        # the saved state: past the global-step start-up where there is one
        s.load_state(state["Q0"])
        if opt.get("t_switch"):
            t = torch.empty(s.n_tris, dtype=torch.int64, device="cuda")
            for _ in range(400):
                s.advance_to(s.t_end, 50)
                s.get_elem_into(t=t)
                if int(t.min()) * s.tick > 0.0099:
                    break
            s.advance_to(s.t_end, 300)
        else:
            s.advance_to(s.t_end, 50)
        state["saved"] = {k: v.cpu().cuda() for k, v in _read(s, _outputs(s)).items()}
        state["nodes"] = tuple(torch.tensor(a, device="cuda") for a in s.get_nodes())
    return state


def _read(s, out):
    s.get_elem_into(**out)
    return out


def run(state):
    s = state["solver"]
    if state["do"] == "adjoint":
        state["Q0"].grad = state["xy0"].grad = None
        Q, X = A.LtsRun.apply(state["Q0"], state["xy0"], s, state["sweeps"], 10)
        A.kinetic_energy(Q, X, state["mask"]).backward()
        return dict(Q=Q, X=X, dQ0=state["Q0"].grad, dxy0=state["xy0"].grad)
    updates = 0
    if state["do"] == "restart":
        s.set_elem(state["saved"])
        s.set_nodes(*state["nodes"])
        s.enqueue(state["sweeps"])
        updates = s.sync()
    else:
        s.load_state(state["Q0"])
        if state["do"] == "advance":
            updates = s.advance_to(state["t_end"], state["sweeps"])[1]
        elif state["do"] == "steps":
            updates = sum(s.sweep() for _ in range(state["sweeps"]))
    return dict(_read(s, state["out"]), updates=updates)


def work(case):
    """FP64 operations of the method (reconstruction, predictor, fluxes per
    update; about 1.2, 5.0 and 17 x 10^4 at order 1, 2, 3) and the state's
    bytes.  How many elements a local step finds ready depends on the data:
    about one in a hundred."""
    n, order, sweeps = case["size"], case["order"], case.get("sweeps", 0)
    per = {1: 1.2e4, 2: 5.0e4, 3: 1.7e5}[order]
    updates = n + sweeps * n * (1.0 if case.get("gts") else 0.01)
    nst = (order + 1) * (order + 1) * (order + 2) // 2
    back = 2.5 if case["do"] == "adjoint" else 0.0
    return dict(bytes=8.0 * n * (4 + 4 + 4 + 3 + 6 + 3 + 4 * nst), flops=updates * per * (1.0 + back))


# ---------------------------------------------------------------------------
# the pre-processing phase in plain 64-bit torch
# ---------------------------------------------------------------------------

def exact(case, seed):
    """The state after the pre-processing phase.  Runs of many local steps and
    their gradients have no evaluation here: the schedule of the steps is part
    of the scheme, and in plain torch they take minutes."""
    if case["do"] != "load":
        return None
    mesh, q, _ = _inputs(case, seed)
    M = case["order"]
    Q = torch.tensor(q)
    X = torch.tensor(W._corner_coords(mesh).reshape(-1, 6))
    w0, dt = _weno(M, mesh, Q, X, 1.4, 0.5)
    tick = 1.0 / 2 ** 20
    ticks = torch.floor(dt / tick).clamp(1, 2 ** 20)
    qhat = _predictor(M, w0, X, ticks * tick, 1.4, case.get("eulerian", False))
    zero = torch.zeros_like(Q)
    return dict(Q=Q, QM=zero, HM=zero[:, :3], X=X, qhat=qhat, t=None, dt=None, count=None, updates=None)


def _exponents(M):
    return [(d - b, b) for d in range(M + 1) for b in range(d + 1)]


def _lattice(M):
    return torch.tensor([(i / M, j / M) for j in range(M + 1) for i in range(M + 1 - j)], dtype=torch.float64)


def _gauss_triangle(n):
    x, w = np.polynomial.legendre.leggauss(n)
    x, w = 0.5 * (x + 1.0), 0.5 * w
    u, v = np.meshgrid(x, x, indexing="ij")
    wt = np.outer(w, w) * (1 - v) * 2.0
    return torch.tensor((u * (1 - v)).ravel()), torch.tensor(v.ravel()), torch.tensor(wt.ravel())


def _mono(x, y, ex, da=0, db=0):
    """d^(da+db) of x^a y^b, last dimension over the exponents."""
    out = []
    for a, b in ex:
        c = math.perm(a, da) * math.perm(b, db)
        out.append(c * x ** (a - da) * y ** (b - db) if a >= da and b >= db else torch.zeros_like(x))
    return torch.stack(out, -1)


def _stencils(M, tri, X, period, n_e):
    """[n, 7, n_e] members of the seven stencils (-1: none), nearest first."""
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    n = tri.shape[0]
    inc = torch.zeros((n, int(tri.max()) + 1), device=dev)
    inc[torch.arange(n, device=dev)[:, None], tri.to(dev).long()] = 1.0
    adj = ((inc @ inc.T) > 0).float()  # elements with a common vertex
    reach = [adj]
    for _ in range(M + 1):
        reach.append(((reach[-1] @ adj) > 0).float())
    P = X.to(dev).reshape(n, 3, 2)
    cen = (P[:, 0] + P[:, 1] + P[:, 2]) / 3.0
    per = None if period is None else torch.tensor(period, device=dev)
    out = torch.full((n, 7, n_e), -1, dtype=torch.int64, device=dev)
    for lo in range(0, n, 1024):
        rows = torch.arange(lo, min(n, lo + 1024), device=dev)
        D = cen[None] - cen[rows][:, None]
        if per is not None:
            D = D - torch.floor(D / per + 0.5) * per
        d2 = D[..., 0] * D[..., 0] + D[..., 1] * D[..., 1]
        own = rows[:, None] == torch.arange(n, device=dev)[None]
        masks = [reach[M][rows] > 0]
        for s in range(6):
            a, b = P[rows, s % 3] - cen[rows], P[rows, (s + 1) % 3] - cen[rows]
            al = D[..., 0] * b[:, None, 1] - D[..., 1] * b[:, None, 0]
            be = a[:, None, 0] * D[..., 1] - a[:, None, 1] * D[..., 0]
            sgn = -1.0 if s >= 3 else 1.0
            masks.append(((reach[M + 1][rows] > 0) & (sgn * al >= 0) & (sgn * be >= 0)) | own)
        for s, m in enumerate(masks):
            d, j = torch.sort(torch.where(m, d2, math.inf), dim=1, stable=True)
            full = torch.isfinite(d[:, n_e - 1])
            out[rows, s] = torch.where(full[:, None], j[:, :n_e], -1)
    return out.cpu()


def _weno(M, mesh, Q, X, gamma, cfl):
    """Nodal values [n, nodes, 4] of the limited polynomials and the local steps."""
    ex = _exponents(M)[1:]
    n, n_e = Q.shape[0], (M + 1) * (M + 2)
    st = _stencils(M, torch.tensor(mesh["tri"]), X, mesh["period"], n_e)
    P = X.reshape(n, 3, 2)
    J = torch.stack([P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]], -1)
    Ji = torch.linalg.inv(J)
    s, t, w = _gauss_triangle(4)
    mean = (w[:, None] * _mono(s - 1 / 3, t - 1 / 3, ex)).sum(0)
    cen = P.mean(1)
    member = st[:, :, 1:].clamp(min=0)
    V = P[member] - P[:, None, None, None, 0]
    if mesh["period"] is not None:
        per = torch.tensor(mesh["period"])
        V = V - (torch.floor((cen[member] - cen[:, None, None]) / per + 0.5) * per)[:, :, :, None]
    R = torch.einsum("nab,nsmkb->nsmka", Ji, V)
    xi = R[..., 0, 0, None] * (1 - s - t) + R[..., 1, 0, None] * s + R[..., 2, 0, None] * t
    et = R[..., 0, 1, None] * (1 - s - t) + R[..., 1, 1, None] * s + R[..., 2, 1, None] * t
    rows = (w[:, None] * _mono(xi - 1 / 3, et - 1 / 3, ex)).sum(-2) - mean
    rhs = Q[member] - Q[:, None, None]
    scale = rows.norm(dim=-2, keepdim=True)
    q_, r_ = torch.linalg.qr(rows / scale)
    C = torch.linalg.solve_triangular(r_, q_.transpose(-1, -2) @ rhs, upper=True) / scale.transpose(-1, -2)
    # characteristic fields along the central polynomial's density gradient
    g = torch.einsum("na,nab->nb", C[:, 0, :2, 0], Ji)
    gn = g.norm(dim=1, keepdim=True)
    nrm = torch.where(gn > 0, g / gn, torch.tensor([1.0, 0.0], dtype=torch.float64))
    nx, ny = nrm[:, 0], nrm[:, 1]
    rho, u, v = Q[:, 0], Q[:, 1] / Q[:, 0], Q[:, 2] / Q[:, 0]
    p = (gamma - 1) * (Q[:, 3] - 0.5 * rho * (u * u + v * v))
    a, H = torch.sqrt(gamma * p / rho), (Q[:, 3] + p) / rho
    un, ut = u * nx + v * ny, v * nx - u * ny
    one, nil = torch.ones_like(u), torch.zeros_like(u)
    Rm = torch.stack([torch.stack([one, one, nil, one], -1), torch.stack([u - a * nx, u, -ny, u + a * nx], -1),
                      torch.stack([v - a * ny, v, nx, v + a * ny], -1),
                      torch.stack([H - a * un, 0.5 * (u * u + v * v), ut, H + a * un], -1)], 1)
    ch = C @ torch.linalg.inv(Rm)[:, None].transpose(-1, -2)
    S = torch.zeros((len(ex), len(ex)), dtype=torch.float64)
    for da in range(M + 1):
        for db in range(M + 1 - da):
            if da + db:
                m = _mono(s - 1 / 3, t - 1 / 3, ex, da, db)
                S += 0.5 * torch.einsum("q,qa,qb->ab", w, m, m)
    sig = torch.einsum("nsav,ab,nsbv->nsv", ch, S, ch)
    lam = torch.ones(7, dtype=torch.float64)
    lam[0] = 1e5
    om = torch.where(st[:, :, :1] >= 0, lam[None, :, None] / (sig + 1e-14) ** 8, 0.0)
    om = om / om.sum(1, keepdim=True)
    coef = torch.einsum("nsv,nsav->nav", om, torch.where(st[:, :, :1, None] >= 0, ch, 0.0)) @ Rm.transpose(-1, -2)
    lat = _lattice(M)
    nodal = Q[:, None] + (_mono(lat[:, 0] - 1 / 3, lat[:, 1] - 1 / 3, ex) - mean) @ coef
    # positivity scaling: density, then pressure through its chord bound
    lo = 1e-8 * rho
    th = torch.where(nodal[:, :, 0] < lo[:, None], (rho - lo)[:, None] / (rho[:, None] - nodal[:, :, 0]), 1.0).amin(1)
    nodal = torch.where((th < 1)[:, None, None], Q[:, None] + th[:, None, None] * (nodal - Q[:, None]), nodal)
    pn = (gamma - 1) * (nodal[..., 3] - 0.5 * (nodal[..., 1] ** 2 + nodal[..., 2] ** 2) / nodal[..., 0])
    th = torch.where(pn < 1e-8 * p[:, None], (p * (1 - 1e-8))[:, None] / (p[:, None] - pn), 1.0).amin(1)
    nodal = torch.where((th < 1)[:, None, None], Q[:, None] + th[:, None, None] * (nodal - Q[:, None]), nodal)
    # local step: incircle diameter over |v| + c of the element and its edge neighbours
    E = P[:, [1, 2, 0]] - P
    dia = 2.0 * torch.linalg.det(J) / E.norm(dim=2).sum(1)
    step = cfl * dia / (torch.sqrt(u * u + v * v) + a)
    edge = {}
    for i, tr in enumerate(mesh["tri"].tolist()):
        for e in range(3):
            edge[(tr[e], tr[(e + 1) % 3])] = i
    dt = step.clone()
    nb = torch.tensor([[edge.get((tr[(e + 1) % 3], tr[e]), i) for e in range(3)]
                       for i, tr in enumerate(mesh["tri"].tolist())])
    return nodal, torch.minimum(dt, step[nb].amin(1))


def _predictor(M, w0, X, dt, gamma, eulerian):
    """[n, (M+1) * nodes, 4]: M + 1 Picard iterations of the space-time Galerkin predictor."""
    lat, ex = _lattice(M), _exponents(M)
    Vi = torch.linalg.inv(_mono(lat[:, 0], lat[:, 1], ex))
    Dx, De = _mono(lat[:, 0], lat[:, 1], ex, 1, 0) @ Vi, _mono(lat[:, 0], lat[:, 1], ex, 0, 1) @ Vi
    h = {1: [], 2: [0.5], 3: [0.5 - math.sqrt(5) / 10, 0.5 + math.sqrt(5) / 10]}[M]
    tau = torch.tensor([0.0] + h + [1.0], dtype=torch.float64)
    k = torch.arange(M + 1, dtype=torch.float64)
    Li = torch.linalg.inv(tau[:, None] ** k)
    x, w = np.polynomial.legendre.leggauss(M + 2)
    x, w = torch.tensor(0.5 * (x + 1)), torch.tensor(0.5 * w)
    L = x[:, None] ** k @ Li
    dL = (k * x[:, None] ** (k - 1).clamp(min=0)) @ Li
    Dt = (k * tau[:, None] ** (k - 1).clamp(min=0)) @ Li
    K, Mm = L.T @ (w[:, None] * dL), L.T @ (w[:, None] * L)
    B = torch.linalg.solve(K[1:, 1:], Mm[1:])
    P = X.reshape(-1, 3, 2)
    pos0 = P[:, None, 0] + lat[None, :, :1] * (P[:, 1] - P[:, 0])[:, None] + \
        lat[None, :, 1:] * (P[:, 2] - P[:, 0])[:, None]
    q, pos = w0[:, None].repeat(1, M + 1, 1, 1), pos0[:, None].repeat(1, M + 1, 1, 1)
    for _ in range(M + 1):
        u, v = q[..., 1] / q[..., 0], q[..., 2] / q[..., 0]
        p = (gamma - 1) * (q[..., 3] - 0.5 * q[..., 0] * (u * u + v * v))
        f = torch.stack([q[..., 1], q[..., 1] * u + p, q[..., 1] * v, u * (q[..., 3] + p)], -1)
        g = torch.stack([q[..., 2], q[..., 2] * u, q[..., 2] * v + p, v * (q[..., 3] + p)], -1)
        vel = torch.stack([u, v], -1) * (0.0 if eulerian else 1.0)
        dx = lambda z: torch.einsum("rs,nts...->ntr...", Dx, z)  # noqa: E731
        de = lambda z: torch.einsum("rs,nts...->ntr...", De, z)  # noqa: E731
        px, pe = dx(pos), de(pos)
        pt = torch.einsum("tu,nus...->nts...", Dt, pos) / dt[:, None, None, None]
        det = px[..., 0] * pe[..., 1] - pe[..., 0] * px[..., 1]
        xix, xiy, etx, ety = pe[..., 1] / det, -pe[..., 0] / det, -px[..., 1] / det, px[..., 0] / det
        xit, ett = -(xix * pt[..., 0] + xiy * pt[..., 1]), -(etx * pt[..., 0] + ety * pt[..., 1])
        rhs = -(dx(f) * xix[..., None] + de(f) * etx[..., None] + dx(g) * xiy[..., None] + de(g) * ety[..., None]
                + dx(q) * xit[..., None] + de(q) * ett[..., None])
        up = lambda z: torch.einsum("tu,nus...->nts...", B, z) * dt[:, None, None, None]  # noqa: E731
        qn, pn = w0[:, None] + up(rhs), pos0[:, None] + up(vel)
        q, pos = torch.cat([w0[:, None], qn], 1), torch.cat([pos0[:, None], pn], 1)
    p = (gamma - 1) * (q[..., 3] - 0.5 * (q[..., 1] ** 2 + q[..., 2] ** 2) / q[..., 0])
    bad = ((q[..., 0] <= 0) | (p <= 0)).flatten(1).any(1)
    q = torch.where(bad[:, None, None, None], w0[:, None].expand_as(q), q)
    return q.flatten(1, 2)
