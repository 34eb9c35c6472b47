"""The coarsest grid's dense product by mirror classes, on grids with and
without cells or nodes on the mirror lines (even and odd sizes), against a direct
solve of the oracle's velocity block and against the cluster launch, which takes
the full inverse."""
import numpy as np
import pytest
import scipy.sparse as sp
import scipy.sparse.linalg as spl

import fsi_inputs as fi
from gpu_helpers import rel
from oracle import fsi_oracle as fo

pytestmark = pytest.mark.gpu


def _case(N):
    xy, tris = fi.ring_disk_mesh(3, 0.2, (0.47, 0.52))
    return fi.FsiCase(N=N, rho_f=1.3, nu=0.05, kappa=30.0, dt=0.005, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 7, lid_u=1.0), X0=xy.copy())


@pytest.mark.parametrize("N", [2, 4, 6, 10, 12, 14, 16])
def test_single_level_velocity_is_the_direct_solve(N):
    """Up to 16 cells the grid is its own coarsest one, so the block-diagonal
    preconditioner's velocity part is A_f^-1 v.  FP64: 1e-11 as the inverse's own
    test; FP32: 1e-5."""
    from paper_2301_10041_gb300 import fsi
    case = _case(N)
    grid = fo.FluidGrid(N)
    M, K, _ = fo.assemble_fluid(grid, case.nu)
    A = (case.rho_f / case.dt * M + K).tocsr()[grid.interior_dofs][:, grid.interior_dofs]
    g = fsi.problem_from_case(case, precision=1, precond=0, restart=10)
    try:
        g.assemble_step()
        rank = np.searchsorted(grid.interior_nodes, g.interior_nodes())
        q = (2 * rank[:, None] + np.arange(2)).ravel()      # library order from the oracle's
        v = np.zeros(g.n)
        f = np.random.default_rng(N).standard_normal(g.n_u)
        v[:g.n_u] = f[q]
        ref = spl.spsolve(sp.csc_matrix(A), f)[q]
        # the pressure part of v is zero, so the velocity part is A_f^-1 v_u alone
        assert rel(g.apply_preconditioner(v, precision=0)[:g.n_u], ref) < 1e-11
        assert rel(g.apply_preconditioner(v, precision=1)[:g.n_u], ref) < 1e-5
    finally:
        g.close()


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N,mg_coarse", [(20, 8), (40, 8), (24, 6), (28, 7), (32, 8)])   # coarsest 5, 5, 6, 7, 8 cells
def test_classes_match_the_full_inverse(N, mg_coarse, precision):
    from paper_2301_10041_gb300 import fsi
    case = _case(N)
    kw = dict(precision=precision, precond=2, stokes_its=2, restart=10, mg_fused=-1, mg_coarse=mg_coarse)
    full = fsi.problem_from_case(case, mg_cluster=0, **kw)
    cls = fsi.problem_from_case(case, mg_cluster=-1, **kw)
    try:
        full.assemble_step()
        cls.assemble_step()
        v = np.random.default_rng(5).standard_normal(full.n)
        for p in sorted({0, precision}):
            assert rel(full.apply_preconditioner(v, precision=p), cls.apply_preconditioner(v, precision=p)) < (
                1e-12 if p == 0 else 2e-5)
    finally:
        full.close()
        cls.close()
