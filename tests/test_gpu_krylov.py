"""Gram-Schmidt, Givens and least-squares kernels of the FP64 solve at the
sizes where they can go wrong: few and many basis vectors (one and several
groups of 32 per warp), a ragged last chunk of rows, and both chunk sizes.

When one Arnoldi cycle stops, its residual estimate says the target is met;
the next cycle's true FP64 residual confirms it only if the basis is
orthonormal, the rotations and the triangular solve are right, and the update
is applied.  So a solve within one cycle reports no restart, and its residual
can be recomputed from the operator and right-hand side on the host."""
import numpy as np
import pytest

import fsi_inputs as fi

pytestmark = pytest.mark.gpu


def _case(N, kappa, nu, dt, seed=5):
    xy, tris = fi.ring_disk_mesh(max(4, int(0.4 * N)), 0.2, (0.5, 0.5))
    return fi.FsiCase(N=N, rho_f=1.0, nu=nu, kappa=kappa, dt=dt, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, seed, lid_u=1.0), X0=xy.copy(), precond=1)


def _pack(prob, u, p, X, lam):
    return np.concatenate([u[prob.interior_nodes()].ravel(), p.ravel(), X.ravel(), lam.ravel()])


@pytest.mark.parametrize("N,kappa,nu,dt,stokes_its,least", [
    (16, 10.0, 1.0, 1e-2, 1, 2),        # one group of vectors
    (20, 300.0, 0.02, 1e-3, 1, 33),     # several groups, n no multiple of the chunk
    (32, 100.0, 0.1, 1e-3, 1, 2),
    (48, 10.0, 0.1, 1e-2, 1, 2),
    (224, 10.0, 0.1, 1e-3, 2, 2),       # more than 2^19 unknowns: the larger chunk
])
def test_one_cycle_reaches_its_estimate(N, kappa, nu, dt, stokes_its, least):
    from paper_2301_10041_gb300 import fsi
    case = _case(N, kappa, nu, dt)
    g = fsi.problem_from_case(case, precision=0, precond=1, rtol=1e-9, stokes_its=stokes_its, restart=250)
    try:
        g.assemble_step()
        info = g.solve_step()
        assert least <= info.iterations < 250
        assert info.restarts == 0 and info.rel_residual <= 1e-9
        x = _pack(g, *g.get_state())
        b = g.get_rhs()
        r = b - g.apply_operator(x, precision=0)
        # the same residual up to the rounding of A x (|A||x| is at most some 1e3 |b| here)
        assert np.linalg.norm(r) <= (1e-9 + 1e-12) * np.linalg.norm(b)
    finally:
        g.close()
