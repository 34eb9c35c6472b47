"""The two routes of the orthogonalisation at their edges: the cluster launch just
below its row limits (4096 unknowns in FP64, 8192 in mixed precision) and the separate
launches just above them, and the separate launches with more than 32 basis vectors
at both chunk sizes (the second trip of their loops over groups of vectors, the
eight-column updates).  The route shows in the launches of an iteration: the cluster
is one, the separate passes and the basis vector are four.

As in the tests of the kernels: an Arnoldi cycle's estimate is confirmed by the next
cycle's true residual only if the basis is orthonormal, the rotations are right and
the update is applied; so a FP64 solve within one cycle reports no restart, and the
residual can be formed from the operator and right-hand side on the host."""
import numpy as np
import pytest

import fsi_inputs as fi

pytestmark = pytest.mark.gpu


def _problem(N, rings, kappa, nu, dt, precision):
    from paper_2301_10041_gb300 import fsi
    xy, tris = fi.ring_disk_mesh(rings, 0.2, (0.5, 0.5))
    case = fi.FsiCase(N=N, rho_f=1.0, nu=nu, kappa=kappa, dt=dt, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 5, lid_u=1.0), X0=xy.copy(), precond=1)
    return fsi.problem_from_case(case, precision=precision, precond=1, rtol=1e-9, restart=250)


def _solve(g, least):
    g.assemble_step()
    info = g.solve_step()
    assert least <= info.iterations < 250
    assert info.rel_residual <= 1e-9
    u, p, X, lam = g.get_state()
    x = np.concatenate([u[g.interior_nodes()].ravel(), p.ravel(), X.ravel(), lam.ravel()])
    b = g.get_rhs()
    r = b - g.apply_operator(x, precision=0)
    # the same residual up to the rounding of A x (|A||x| is at most some 1e3 |b| here)
    assert np.linalg.norm(r) <= (1e-9 + 1e-12) * np.linalg.norm(b)
    return info


@pytest.mark.parametrize("N,limit,rings,precision", [(16, 4096, (10, 11), 0), (24, 8192, (12, 13), 1)])
def test_cluster_limit(N, limit, rings, precision):
    below = _problem(N, rings[0], 300.0, 0.02, 1e-3, precision)
    above = _problem(N, rings[1], 300.0, 0.02, 1e-3, precision)
    try:
        assert limit - 256 < below.n <= limit < above.n < limit + 256
        assert above.graph_kernel_counts()[3] == below.graph_kernel_counts()[3] + 3
        for g in (below, above):
            info = _solve(g, 33)
            assert precision == 1 or info.restarts == 0
    finally:
        below.close()
        above.close()


@pytest.mark.parametrize("N,rings,kappa,nu", [
    (48, 19, 300.0, 0.02),      # up to 2^19 unknowns: the smaller chunk
    (224, 89, 100.0, 0.05),     # beyond: the larger one
])
def test_many_vectors_of_the_separate_launches(N, rings, kappa, nu):
    g = _problem(N, rings, kappa, nu, 1e-3, 0)
    try:
        assert g.n > 16384 and (g.n > 2 ** 19) == (N == 224)
        assert _solve(g, 33).restarts == 0
    finally:
        g.close()
