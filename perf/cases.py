"""Timed cases of the FSI library: whole time steps, batches of instances, one
Krylov iteration's products and the allocation-free point location, each
through the public binding (``paper_2301_10041_gb300.fsi``).

A step case is what a time-stepping program does for one step of one
instance: ``set_state`` (the step's u^n and X^n, host arrays), ``step``
(assembly of C_f(X^n), the linear solve, advance) and ``get_state``.  Two
settings recur:

* the block-triangular preconditioner (the default and the paper's better
  one), with one V-cycle pair per application or with 8 Richardson steps on
  the Stokes block (the stiff workloads);
* tolerances of 1e-10 to 1e-12 as in the 16 x 16 single-step workload and the
  parity tests, so that a returned state is the discrete solution and not the
  place where the iteration happened to stop.

Sizes and materials are those of ``fsi_inputs`` and the benchmark's
workloads.  Initial velocities are uniform per dof and bodies slightly
stretched and turned, both drawn from the seed.
"""
import math

import numpy as np
import torch

import fsi_inputs as fi
from paper_2301_10041_gb300 import fsi


def _step(name, **kw):
    """A step of one instance; kw overrides the served workload's defaults."""
    c = dict(kind="step", N=64, body="disk", R=0.2, cx=0.5, cy=0.5, rings=0, nu=0.1, kappa=100.0, dt=1e-3, lid=1.0,
             amplitude=1.0, precision=1, precond=1, stokes_its=8, restart=60, inner_rtol=0.0, rtol=1e-11, coupling=0)
    c.update(kw)
    if name:
        c["name"] = name
    return c


def listed():
    return [
        # the plain method: FP64, block-diagonal, the 16 x 16 cavity with the 216-triangle disk (the smoke step)
        _step("plain_fp64_16", N=16, rings=6, nu=1.0, kappa=10.0, dt=1e-2, lid=0.0, precision=0, precond=0,
              stokes_its=1, restart=200, rtol=1e-12),
        # a small instance whose grid is no power of two, one V-cycle pair per application: launch latency
        _step("small_mixed_24", N=24, R=0.17, cx=0.45, cy=0.55, dt=1e-2, kappa=10.0, stokes_its=1),
        # an ordinary served request: ellipse under a lid, mixed precision
        _step("served_mixed_64", N=64, body="ellipse", R=0.22),
        # the 128 x 128 lid-driven cavity with the stiff disk, mixed precision: the benchmark's flagship workload
        _step("cavity_mixed_128", N=128, rings=36, nu=0.01, kappa=1e3, restart=30, inner_rtol=1e-4, rtol=1e-10),
        # the same grid in FP64 throughout, the arm the mixed one is compared with
        _step("cavity_fp64_128", N=128, rings=36, restart=100, precision=0),
        # size sweep, one V-cycle pair per application, C_f by mesh intersection (the paper's own rule)
        _step("sweep_exact_256", N=256, body="ellipse", rings=103, kappa=10.0, dt=1e-2, stokes_its=1, restart=100,
              rtol=1e-10, coupling=1),
        # size sweep, the largest step of the list
        _step("sweep_mixed_512", N=512, body="ellipse", rings=205, rtol=1e-10),
        # the paper's linear test: quarter annulus with the Q1 solid, released from the stretched state
        dict(kind="annulus", name="annulus_q1_112", N=112, quads=True, precision=1, stokes_its=1, restart=100,
             rtol=1e-11),
        # the paper's nonlinear test: the bar with the exponential law, Newton around the linear solves
        dict(kind="bar", name="bar_newton_64", N=64, nx=32, ny=8, precision=1, stokes_its=1, restart=60, rtol=1e-12),
        # uneven instances stepped together, each on its own stream
        dict(kind="batch", name="batch_12", count=12, first=0, rtol=1e-11),
        # one iteration of an outer Krylov method: z = P^-1 v and y = A x in FP32 at the benchmark's settings
        dict(kind="krylov", name="krylov_128", N=128, rings=36, nu=0.01, kappa=1e3, dt=1e-3, precond=2, stokes_its=8),
        # point location and binning for callers that may not allocate
        dict(kind="locate", name="locate_bin_256", N=256, rings=103),
    ]


#: grids the library takes, up to the size sweep's second largest: c 2^k with c <= 8
GRIDS = (16, 20, 24, 28, 32, 40, 48, 56, 64, 80, 96, 112, 128, 160, 192, 224, 256, 320)


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(("step",) * 7 + ("annulus", "bar", "batch", "krylov", "locate"))
    if kind == "annulus":
        return dict(kind=kind, N=rng.choice((24, 40, 48, 64, 96, 128, 160)), quads=rng.random() < 0.5, precision=1,
                    stokes_its=1, restart=100, rtol=1e-11)
    if kind == "bar":
        N = rng.choice((24, 32, 48, 64, 96))
        return dict(kind=kind, N=N, nx=N // 2 + rng.randrange(3), ny=N // 8 + rng.randrange(2), precision=1,
                    stokes_its=1, restart=60, rtol=1e-12)
    if kind == "batch":
        return dict(kind=kind, count=rng.randrange(3, 15), first=rng.randrange(0, 200), rtol=1e-11)
    if kind == "krylov":
        N = rng.choice((32, 48, 64, 112, 128, 192, 256))
        return dict(kind=kind, N=N, rings=max(6, int(0.28 * N)), nu=_log(rng, 0.01, 1.0), kappa=_log(rng, 10.0, 1e3),
                    dt=rng.choice((1e-3, 1e-2)), precond=rng.choice((0, 1, 2, 3)), stokes_its=rng.choice((1, 2, 4, 8)))
    if kind == "locate":
        N = int(_log(rng, 16, 512))
        return dict(kind=kind, N=N, rings=max(4, int(0.4 * N * rng.uniform(0.7, 1.2))))
    fp64 = rng.random() < 0.25
    N = rng.choice([n for n in GRIDS if n <= (128 if fp64 else 320)])
    return _step("", N=N, body=rng.choice(("disk", "ellipse")), R=rng.uniform(0.1, 0.25), cx=rng.uniform(0.4, 0.6),
                 cy=rng.uniform(0.4, 0.6), nu=_log(rng, 0.05, 0.3), kappa=_log(rng, 1.0, 100.0),
                 dt=rng.choice((1e-3, 1e-2)), lid=float(rng.randrange(2)), precision=0 if fp64 else 1,
                 precond=rng.choice((0, 1, 1, 1)), stokes_its=rng.choice((1, 1, 4, 8)),
                 restart=rng.choice((60, 100)), rtol=1e-11 if N <= 128 else 1e-10, coupling=int(rng.random() < 0.2))


# ------------------------------------------------------------------- inputs
def _moved(xy, seed):
    """The body's positions X^n: the reference mesh turned by up to 0.1 rad
    about its centre and stretched by up to 3 %, area kept."""
    r = fi.uniform01(seed * 977 + 13, np.arange(2))
    th, s = 0.2 * (r[0] - 0.5), 1.0 + 0.06 * (r[1] - 0.5)
    c = xy.mean(axis=0)
    d = (xy - c) * np.array([s, 1.0 / s])
    return c + d @ np.array([[math.cos(th), math.sin(th)], [-math.sin(th), math.cos(th)]])


def _disk_or_ellipse(case):
    m = case["rings"] or int(math.ceil(2.0 * case["R"] * case["N"]))
    if case["body"] == "ellipse":
        return fi.ellipse_mesh(m, case["R"], 0.5 * case["R"], 30.0, (case["cx"], case["cy"]))
    return fi.ring_disk_mesh(m, case["R"], (case["cx"], case["cy"]))


def _fsi_case(case, seed):
    if case["kind"] == "annulus":
        c = fi.annulus_case(case["N"], quads=case["quads"])
        c.u0 = fi.initial_velocity(c.N, seed, amplitude=0.2)
        return c
    if case["kind"] == "bar":
        c = fi.bar_case(case["N"], case["nx"], case["ny"])
        c.u0 = fi.initial_velocity(c.N, seed, amplitude=0.1)
        return c
    xy, tris = _disk_or_ellipse(case)
    return fi.FsiCase(N=case["N"], rho_f=1.0, nu=case["nu"], kappa=case["kappa"], dt=case["dt"], lid_u=case["lid"],
                      ref_xy=xy, tris=tris, u0=fi.initial_velocity(case["N"], seed, case["lid"], case["amplitude"]),
                      X0=_moved(xy, seed))


def _batch_cases(case, seed):
    """Instances of the uneven batch (sizes, radii, centres, viscosities by
    ``batch_instance``), with kappa = 1 .. 100 and nu >= 0.05."""
    out = []
    for i in range(case["first"], case["first"] + case["count"]):
        c = fi.batch_instance(i)
        c.u0 = fi.initial_velocity(c.N, seed * 1009 + i)
        c.X0 = _moved(c.ref_xy, seed + i)
        c.kappa = math.sqrt(c.kappa)
        c.nu = max(c.nu, 0.05)
        out.append(c)
    return out


def _problem(c, case):
    extra = {"inner_rtol": case["inner_rtol"]} if case.get("inner_rtol") else {}
    return fsi.problem_from_case(c, precision=case["precision"], precond=case.get("precond", 1), rtol=case["rtol"],
                                 stokes_its=case["stokes_its"], restart=case["restart"], max_it=4000,
                                 coupling=case.get("coupling", 0), **extra)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        cs = _batch_cases(case, seed)
        probs = [fsi.problem_from_case(c, precision=1, precond=1, rtol=case["rtol"], stokes_its=8, restart=60,
                                       max_it=4000) for c in cs]
        return {"kind": kind, "cases": cs, "problems": probs}
    if kind == "krylov":
        full = _step("", **{k: v for k, v in case.items() if k not in ("kind", "name")})
        c = _fsi_case(full, seed)
        p = _problem(c, full)
        p.assemble_step()
        r = np.random.default_rng(seed)
        v = r.standard_normal(p.n)
        v[p.n_u:p.n_u + p.n_p:3] -= v[p.n_u:p.n_u + p.n_p:3].mean()
        return {"kind": kind, "problem": p, "v": v / np.linalg.norm(v), "x": r.standard_normal(p.n)}
    if kind == "locate":
        xy, tris = fi.ellipse_mesh(case["rings"], 0.2, 0.1, 30.0)
        X = torch.as_tensor(_moved(xy, seed)).cuda()
        npts, cells = 6 * len(tris), case["N"] * case["N"]
        ints = dict(dtype=torch.int32, device="cuda")
        return {"kind": kind, "N": case["N"], "n_tris": len(tris), "tris": torch.as_tensor(tris).cuda(), "X": X,
                "cell": torch.zeros(npts, **ints), "xi": torch.zeros(npts, dtype=torch.float64, device="cuda"),
                "eta": torch.zeros(npts, dtype=torch.float64, device="cuda"), "start": torch.zeros(cells + 1, **ints),
                "points": torch.zeros(npts, **ints), "outside": torch.zeros(1, **ints)}
    c = _fsi_case(case, seed)
    return {"kind": kind, "case": c, "problem": _problem(c, case)}


def _state(p):
    u, pr, X, lam = p.get_state()
    return {"u": u, "p": pr, "X": X, "lam": lam}


def run(state):
    kind = state["kind"]
    if kind == "batch":
        for p, c in zip(state["problems"], state["cases"]):
            p.set_state(c.u0, c.X0)
        st, _ = fsi.step_batch(state["problems"])
        if st != fsi.FSI_OK:
            raise fsi.FsiError(st, "fsi_step_batch")
        return [_state(p) for p in state["problems"]]
    if kind == "krylov":
        p = state["problem"]
        # both products are FP32 values in the library; the ABI hands them over as doubles
        z = p.apply_preconditioner(state["v"], precision=1).astype(np.float32)
        y = p.apply_operator(state["x"], precision=1).astype(np.float32)
        ends = np.cumsum([p.n_u, p.n_p, p.n_x])      # u | p | X | lambda
        return {"z": np.split(z, ends), "y": np.split(y, ends)}
    if kind == "locate":
        s = state
        st = fsi.locate_bin_noalloc(s["N"], s["n_tris"], s["tris"].data_ptr(), s["X"].data_ptr(), s["cell"].data_ptr(),
                                    s["xi"].data_ptr(), s["eta"].data_ptr(), s["start"].data_ptr(),
                                    s["points"].data_ptr(), s["outside"].data_ptr(),
                                    torch.cuda.current_stream().cuda_stream)
        if st != fsi.FSI_OK:
            raise fsi.FsiError(st, "fsi_locate_bin_noalloc")
        return {k: s[k] for k in ("cell", "xi", "eta", "start", "points", "outside")}
    p, c = state["problem"], state["case"]
    p.set_state(c.u0, c.X0)
    p.step()
    return _state(p)


# --------------------------------------------------------------------- work
def _solid_nodes(case):
    m = case.get("rings") or int(math.ceil(2.0 * case.get("R", 0.2) * case["N"]))
    return 1 + 3 * m * (m + 1)


def _step_work(N, ns, stokes_its):
    """One step, whatever the method: the state in and out once, and one
    application of the operator and of the preconditioner (a Krylov solve
    needs at least one): about 64 multiply-adds per Q2 node and 81 per
    pressure cell for each application, 5 per level of a V-cycle, levels
    adding up to 4/3 of the finest."""
    unknowns = 2 * (2 * N - 1) ** 2 + 3 * N * N + 4 * ns
    state_in = 2 * (2 * N + 1) ** 2 + 2 * ns
    op = 256 * N * N + 108 * N * N + 100 * ns
    pair = (5 * 256 + 5 * 81) * N * N * 4 / 3 + 108 * N * N
    return {"bytes": 8.0 * (state_in + unknowns), "flops": 2.0 * (op + stokes_its * pair)}


def work(case):
    kind = case["kind"]
    if kind == "batch":
        w = [_step_work(c.N, len(c.ref_xy), 8) for c in _batch_cases(case, 1)]
        return {"bytes": sum(x["bytes"] for x in w), "flops": sum(x["flops"] for x in w)}
    if kind == "locate":
        m = case["rings"]
        tris, nodes = 6 * m * m, 1 + 3 * m * (m + 1)
        return {"bytes": 12.0 * tris + 16.0 * nodes + 6.0 * tris * 24 + 4.0 * case["N"] ** 2, "flops": 6.0 * tris * 14}
    if kind == "krylov":
        w = _step_work(case["N"], _solid_nodes(case), case["stokes_its"])
        return {"bytes": 2 * w["bytes"], "flops": w["flops"]}
    if kind == "annulus":
        ns = int(0.2 * case["N"] + 1) * int(0.2 * math.pi * case["N"] + 1)
    elif kind == "bar":
        ns = (case["nx"] + 1) * (case["ny"] + 1)
    else:
        ns = _solid_nodes(case)
    return _step_work(case["N"], ns, case["stokes_its"])


# ---------------------------------------------------- the same in 64 bits
# degree-4 rule on the triangle (Dunavant 1985): two orbits of three points
_ORBITS = ((0.44594849091596488632, 0.22338158967801146570), (0.091576213509770743460, 0.10995174365532186764))


def _triangle_rule():
    lam, w = [], []
    for a, wt in _ORBITS:
        for k in range(3):
            p = [a, a, a]
            p[k] = 1.0 - 2.0 * a
            lam.append(p)
            w.append(wt)
    return np.array(lam), np.array(w)


def _quadratics(t):
    return np.stack([(1 - t) * (1 - 2 * t), 4 * t * (1 - t), t * (2 * t - 1)], -1)


def _rule_points(X, tris):
    lam, _ = _triangle_rule()
    P0, P1, P2 = (X[tris[:, k]][:, None, :] for k in range(3))
    return ((P0 + lam[None, :, 1, None] * (P1 - P0)) + lam[None, :, 2, None] * (P2 - P0)).reshape(-1, 2)


def _locate(x, N):
    t = x * N
    i = np.minimum(np.floor(t).astype(np.int64), N - 1)
    return i, t - i


def _dense_step(c):
    """The block system of one step (P1 solid, point rule, linear law)
    assembled densely and solved by LU with refinement: u, p, X, lambda."""
    N, h, n1 = c.N, 1.0 / c.N, 2 * c.N + 1
    r = 0.5 * math.sqrt(0.6)
    g, gw = np.array([0.5 - r, 0.5, 0.5 + r]), np.array([5.0, 8.0, 5.0]) / 18.0
    L = _quadratics(g)                                                      # [point, node]
    D = np.stack([4 * g - 3, 4 - 8 * g, 4 * g - 1], -1) / h
    W = (gw[:, None] * gw[None, :] * h * h).ravel()                         # point = (qy, qx)
    val = np.einsum("yb,xa->yxba", L, L).reshape(9, 9)
    gx = np.einsum("yb,xa->yxba", L, D).reshape(9, 9)
    gy = np.einsum("yb,xa->yxba", D, L).reshape(9, 9)
    psi = np.stack([np.ones(9), np.tile(g - 0.5, 3), np.repeat(g - 0.5, 3)], -1)
    ip = lambda a, b: np.einsum("q,qi,qj->ij", W, a, b)                     # noqa: E731
    Me = ip(val, val)
    Ke = np.zeros((9, 2, 9, 2))
    Ke[:, 0, :, 0] = c.nu * (ip(gx, gx) + 0.5 * ip(gy, gy))
    Ke[:, 1, :, 1] = c.nu * (ip(gy, gy) + 0.5 * ip(gx, gx))
    Ke[:, 0, :, 1] = 0.5 * c.nu * ip(gy, gx)
    Ke[:, 1, :, 0] = 0.5 * c.nu * ip(gx, gy)
    Ae = Ke.copy()
    for k in range(2):
        Ae[:, k, :, k] += c.rho_f / c.dt * Me
    Be = np.stack([ip(psi, gx), ip(psi, gy)], -1).reshape(3, 18)            # (div phi, psi)
    cy, cx = np.divmod(np.arange(N * N), N)
    nodes = (2 * cy[:, None] + np.repeat(np.arange(3), 3)) * n1 + 2 * cx[:, None] + np.tile(np.arange(3), 3)
    dofs = (2 * nodes[:, :, None] + np.arange(2)).reshape(N * N, 18)
    nd, npr, ns = 2 * n1 * n1, 3 * N * N, len(c.ref_xy)
    iy, ix = np.divmod(np.arange(n1 * n1), n1)
    inner = np.flatnonzero(np.repeat((ix > 0) & (iy > 0) & (ix < 2 * N) & (iy < 2 * N), 2))
    new = np.full(nd, -1)
    new[inner] = np.arange(inner.size)
    u_wall = fi.wall_velocity(N, c.lid_u).ravel()
    u_n = np.where(new >= 0, np.asarray(c.u0).ravel(), u_wall)
    # solid matrices and C_f by its rule points
    P = c.ref_xy[c.tris]
    d1, d2 = P[:, 1] - P[:, 0], P[:, 2] - P[:, 0]
    det = d1[:, 0] * d2[:, 1] - d1[:, 1] * d2[:, 0]
    g1 = np.stack([d2[:, 1], -d2[:, 0]], -1) / det[:, None]
    g2 = np.stack([-d1[:, 1], d1[:, 0]], -1) / det[:, None]
    G = np.stack([-(g1 + g2), g1, g2], 1)
    Cs, As = np.zeros((ns, ns)), np.zeros((ns, ns))
    ti, tj = np.repeat(c.tris, 3, 1), np.tile(c.tris, (1, 3))
    np.add.at(Cs, (ti, tj), (det / 24)[:, None] * (np.ones((3, 3)) + np.eye(3)).ravel())
    np.add.at(As, (ti, tj), c.kappa * (det / 2)[:, None] * np.einsum("tad,tbd->tab", G, G).reshape(-1, 9))
    lam, w = _triangle_rule()
    cell, loc = _locate(_rule_points(np.asarray(c.X0, dtype=np.float64), c.tris), N)
    phi = np.einsum("pb,pa->pba", _quadratics(loc[:, 1]), _quadratics(loc[:, 0])).reshape(-1, 9)
    pn = nodes[cell[:, 1] * N + cell[:, 0]]
    wq = (0.5 * det[:, None] * w).ravel()
    Cf = np.zeros((ns, n1 * n1))
    for a in range(3):
        np.add.at(Cf, (np.repeat(c.tris[:, a], 6)[:, None], pn), (wq * np.tile(lam[:, a], len(c.tris)))[:, None] * phi)
    # the system over (u inner, p, X, lambda), bordered by the pressure's mean
    nu_, o_p = inner.size, inner.size
    o_x, o_l = o_p + npr, o_p + npr + 2 * ns
    n = o_l + 2 * ns
    A, b = np.zeros((n + 1, n + 1)), np.zeros(n + 1)
    full = np.zeros(n + 1)                                                  # wall data moved to the right
    di, dj = np.repeat(dofs, 18, 1), np.tile(dofs, (1, 18))
    av = np.broadcast_to(Ae.reshape(18, 18).ravel(), di.shape)
    both = (new[di] >= 0) & (new[dj] >= 0)
    np.add.at(A, (new[di[both]], new[dj[both]]), av[both])
    edge = (new[di] >= 0) & (new[dj] < 0)
    np.add.at(full, new[di[edge]], av[edge] * u_wall[dj[edge]])
    m = np.broadcast_to(np.kron(Me, np.eye(2)).ravel(), di.shape)
    rows = new[di] >= 0
    # g1 = (rho/dt) M u^n minus the walls' part of it, which u_D cancels against A_ID u_D's mass part
    np.add.at(b, new[di[rows]], (c.rho_f / c.dt * m * u_n[dj])[rows])
    b[:nu_] -= full[:nu_]
    pr = o_p + 3 * np.arange(N * N)[:, None] + np.repeat(np.arange(3), 18)
    bj = np.tile(dofs, (1, 3))
    bv = np.broadcast_to(Be.ravel(), bj.shape)
    ins = new[bj] >= 0
    np.add.at(A, (pr[ins], new[bj[ins]]), -bv[ins])
    np.add.at(A, (new[bj[ins]], pr[ins]), -bv[ins])
    np.add.at(b, pr[~ins], (bv * u_wall[bj])[~ins])
    C2 = np.kron(Cf, np.eye(2))
    A[o_l:n, :nu_] = C2[:, inner]
    A[:nu_, o_l:n] = C2[:, inner].T
    A[o_x:o_l, o_x:o_l] = np.kron(As, np.eye(2))
    A[o_x:o_l, o_l:n] = -np.kron(Cs, np.eye(2))
    A[o_l:n, o_x:o_l] = -np.kron(Cs, np.eye(2)) / c.dt
    b[o_l:n] = -np.kron(Cs, np.eye(2)) @ np.asarray(c.X0).ravel() / c.dt - C2 @ np.where(new >= 0, 0.0, u_wall)
    A[n, o_p:o_x:3] = A[o_p:o_x:3, n] = 1.0
    s = 1.0 / np.sqrt(np.abs(A).max(axis=1))                                # equilibration
    dev = "cuda" if torch.cuda.is_available() else "cpu"
    S, rhs = torch.as_tensor(A * s[:, None] * s[None, :], device=dev), torch.as_tensor(b * s, device=dev)[:, None]
    lu, piv = torch.linalg.lu_factor(S)
    x = torch.linalg.lu_solve(lu, piv, rhs)
    for _ in range(3):
        x = x + torch.linalg.lu_solve(lu, piv, rhs - S @ x)
    x = x[:, 0].cpu().numpy() * s
    u = u_wall.copy()
    u[inner] = x[:nu_]
    return {"u": u.reshape(-1, 2), "p": x[o_p:o_x].reshape(-1, 3), "X": x[o_x:o_l].reshape(-1, 2),
            "lam": x[o_l:n].reshape(-1, 2)}


def exact(case, seed):
    """Small steps by a dense solve; the location's coordinates by their
    formula.  Larger steps have no solve in plain torch within seconds, and
    the FP32 preconditioner is defined by its own sweeps."""
    if case["kind"] == "locate":
        xy, tris = fi.ellipse_mesh(case["rings"], 0.2, 0.1, 30.0)
        _, loc = _locate(_rule_points(_moved(xy, seed), tris), case["N"])
        return {"cell": None, "xi": loc[:, 0], "eta": loc[:, 1], "start": None, "points": None, "outside": None}
    if case["kind"] == "step" and case["N"] <= 24 and case["coupling"] == 0:
        return _dense_step(_fsi_case(case, seed))
    return None
