"""The solid mass solves of the preconditioner in patches of several Chebyshev
steps per launch, against direct solves with the oracle's solid matrices.

With the block-diagonal preconditioner the solid part is z_X = -dt C_s^-1 v_l,
z_l = C_s^-1 (A_s z_X - v_X), each C_s^-1 by k Chebyshev-Jacobi steps on [1/2, 2]
(P1).  The energy-norm error of k steps is at most 1 / T_k(5/3) =
2 / (3^k + 3^-k) of the solution's energy norm; that bound plus rounding (k steps
of some 20 operations: 1e-12 in FP64, 2e-5 in FP32) is the tolerance.  The degrees
cover one launch and several, the meshes one patch and many, a thin body, and a
fan whose hub row is too wide for patches (the per-step kernels)."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl

import fsi_inputs as fi
from oracle import fsi_oracle as fo

pytestmark = pytest.mark.gpu


def _fan(n=40):
    th = 2 * np.pi * np.arange(n) / n
    xy = np.concatenate([[[0.5, 0.5]], 0.5 + 0.2 * np.stack([np.cos(th), np.sin(th)], 1)])
    return xy, np.array([(0, 1 + i, 1 + (i + 1) % n) for i in range(n)], dtype=np.int32)


MESHES = {
    "disk7": lambda: fi.ring_disk_mesh(1, 0.2, (0.5, 0.5)),
    "disk127": lambda: fi.ring_disk_mesh(6, 0.2, (0.5, 0.5)),
    "disk1141": lambda: fi.ring_disk_mesh(19, 0.2, (0.5, 0.5)),
    "ellipse3997": lambda: fi.ellipse_mesh(36, 0.25, 0.1, 30.0),
    "bar": lambda: fi.bar_mesh(300, 3),
    "fan": _fan,
}


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("degree", [1, 2, 0, 45])
@pytest.mark.parametrize("name", list(MESHES))
def test_mass_solves_meet_the_chebyshev_bound(name, degree, precision):
    from paper_2301_10041_gb300 import fsi
    xy, tris = MESHES[name]()
    dt, kappa = 1e-2, 10.0
    case = fi.FsiCase(N=16, rho_f=1.0, nu=1.0, kappa=kappa, dt=dt, lid_u=0.0, ref_xy=xy, tris=tris,
                      u0=fi.wall_velocity(16, 0.0), X0=xy.copy())
    g = fsi.problem_from_case(case, precision=precision, precond=0, cs_degree=degree, restart=10)
    try:
        g.assemble_step()
        v = np.zeros(g.n)
        rng = np.random.default_rng(3)
        o = g.n_u + g.n_p
        v[o:] = rng.standard_normal(g.n - o)
        z = g.apply_preconditioner(v, precision=precision)
    finally:
        g.close()
    vX, vL = v[o:o + g.n_x].reshape(-1, 2), v[o + g.n_x:].reshape(-1, 2)
    zX, zL = z[o:o + g.n_x].reshape(-1, 2), z[o + g.n_x:].reshape(-1, 2)
    C, A = fo.assemble_solid(xy, tris.astype(np.int64), kappa)
    lu = spl.splu(sp.csc_matrix(C))
    k = degree or (12 if precision else 16)
    tol = 2.0 / (3.0 ** k + 3.0 ** -k) * (1 + 1e-6) + (2e-5 if precision else 1e-12)

    def energy(x):
        return np.sqrt(np.sum(x * (C @ x)))

    for got, rhs in ((zX, -dt * vL), (zL, A @ zX - vX)):
        ref = lu.solve(rhs)
        assert energy(got - ref) <= tol * energy(ref)
