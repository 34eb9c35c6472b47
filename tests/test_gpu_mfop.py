"""The full operator and the Stokes residual without stored matrices, at the
grids where their kernels change: N = 2 (no stencils: sparse kernels), the
smallest with stencils, the smallest FP64 ones, ragged warps (N = 56) and a
power of two.  The reference is the oracle's assembled system; tolerances as in
the operator test of the parity suite (rounding of some 100 products per row)."""
import numpy as np
import pytest

import fsi_inputs as fi
from gpu_helpers import oracle_to_gpu_perm, rel
from oracle import fsi_oracle as fo

pytestmark = pytest.mark.gpu


def _case(N):
    xy, tris = fi.ring_disk_mesh(max(1, N // 8), 0.2, (0.47, 0.52))
    return fi.FsiCase(N=N, rho_f=1.3, nu=0.05, kappa=30.0, dt=0.005, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 7, lid_u=1.0), X0=xy.copy())


@pytest.mark.parametrize("N", [2, 4, 6, 16, 32, 48, 56, 64])
def test_operator_matches_the_assembled_system(N):
    from paper_2301_10041_gb300 import fsi
    case = _case(N)
    o = fo.OracleProblem(case.N, case.rho_f, case.nu, case.kappa, case.dt, case.lid_u, case.ref_xy, case.tris)
    K, rhs, _ = o.system(case.u0, case.X0)
    g = fsi.problem_from_case(case, precision=1, restart=20)
    try:
        g.assemble_step()
        q = oracle_to_gpu_perm(o, g)
        x = np.random.default_rng(3).standard_normal(K.shape[0])
        ref = (K @ x)[q]
        assert rel(g.apply_operator(x[q], precision=0), ref) < 1e-13
        assert rel(g.apply_operator(x[q], precision=1), ref) < 1e-5
        # field by field: a small block must not hide behind a large one
        for a, b in ((0, g.n_u), (g.n_u, g.n_u + g.n_p), (g.n_u + g.n_p, g.n)):
            assert rel(g.apply_operator(x[q], precision=0)[a:b], ref[a:b]) < 1e-12
    finally:
        g.close()


@pytest.mark.parametrize("N", [32, 56])
def test_richardson_steps_take_the_stokes_residual(N):
    """Two Richardson steps against one written out with the operator: with
    P1 one V-cycle pair, z2 = z1 + P1 (r - A_11 z1).  On the FP64 path the
    residual is its own launch; the solid part is left out (v_X = v_l = 0)."""
    from paper_2301_10041_gb300 import fsi
    case = _case(N)
    one = fsi.problem_from_case(case, precision=0, precond=0, stokes_its=1, restart=20)
    two = fsi.problem_from_case(case, precision=0, precond=0, stokes_its=2, restart=20)
    try:
        one.assemble_step()
        two.assemble_step()
        nf = one.n_u + one.n_p
        v = np.zeros(one.n)
        v[:nf] = np.random.default_rng(5).standard_normal(nf)
        z1 = one.apply_preconditioner(v, precision=0)
        r = np.zeros(one.n)
        r[:nf] = (v - one.apply_operator(z1, precision=0))[:nf]
        ref = z1 + one.apply_preconditioner(r, precision=0)
        z2 = two.apply_preconditioner(v, precision=0)
        # rounding of the residual, |A| |z| against |v|: some 1e3 here
        assert rel(z2[:one.n_u], ref[:one.n_u]) < 1e-11
        assert rel(z2[one.n_u:nf], ref[one.n_u:nf]) < 1e-11
    finally:
        one.close()
        two.close()
