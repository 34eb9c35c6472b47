"""mg_fused = -1 keeps the stored sparse matrices throughout: the multigrid
levels, the fluid rows of the full operator and the residual of the Richardson
steps.  It is the assembled form that the matrix-free one is compared with, so it
may not run on the same stencils.  Checked from what the operator reads (the
algorithmic bytes the timing hook reports) and against the oracle's system."""
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


@pytest.mark.parametrize("N,free", [(2, ()), (4, (0,)), (16, (0,)), (64, (0, 1))])   # free: matrix-free by default
def test_operator_reads_the_stored_rows(N, free):
    from paper_2301_10041_gb300 import fsi
    case = _case(N)
    o = fo.OracleProblem(case.N, case.rho_f, case.nu, case.kappa, case.dt, case.lid_u, case.ref_xy, case.tris)
    K, _, _ = o.system(case.u0, case.X0)
    on = fsi.problem_from_case(case, precision=1, restart=20)
    off = fsi.problem_from_case(case, precision=1, restart=20, mg_fused=-1)
    try:
        on.assemble_step()
        off.assemble_step()
        for which, vbytes in ((0, 4), (1, 8)):           # full operator, FP32 and FP64
            more = off.time_kernel(which, 1)[1] - on.time_kernel(which, 1)[1]
            # at least the velocity block: 2 x 2 values and a column per stored
            # block, on average more than nine blocks a row from N = 4 on
            assert (more >= 9 * (on.n_u // 2) * (4 * vbytes + 4)) == (which in free)
            assert which in free or more == 0
        q = oracle_to_gpu_perm(o, off)
        x = np.random.default_rng(3).standard_normal(K.shape[0])
        ref = (K @ x)[q]
        # tolerances as in the operator test of the parity suite
        assert rel(off.apply_operator(x[q], precision=0), ref) < 1e-13
        assert rel(off.apply_operator(x[q], precision=1), ref) < 1e-5
    finally:
        on.close()
        off.close()


@pytest.mark.parametrize("N", [16, 32])
def test_fp32_richardson_residual_matches_the_stored_one(N):
    """The FP32 Stokes residual launch (taken where omega is not 1) on the grid's
    stencils against the one on the stored rows: the same preconditioner up to FP32
    rounding, as the fused levels' own test (2e-5)."""
    from paper_2301_10041_gb300 import fsi
    case = _case(N)
    kw = dict(precision=1, precond=2, stokes_its=3, stokes_omega=0.9, restart=20, mg_cluster=-1)
    on = fsi.problem_from_case(case, **kw)
    off = fsi.problem_from_case(case, mg_fused=-1, **kw)
    try:
        on.assemble_step()
        off.assemble_step()
        v = np.random.default_rng(5).standard_normal(on.n)
        assert rel(on.apply_preconditioner(v, precision=1), off.apply_preconditioner(v, precision=1)) < 2e-5
    finally:
        on.close()
        off.close()


@pytest.mark.parametrize("N,mg_fused,stored", [(16, 0, True), (32, 0, False), (64, 0, False), (64, -1, True)])
def test_fp64_smoothing_step_is_timed_as_it_runs(N, mg_fused, stored):
    """The timing hook's FP64 smoothing step: matrix-free from 32 cells (the six
    vectors and nothing else), on the stored blocks below and with mg_fused = -1."""
    from paper_2301_10041_gb300 import fsi
    g = fsi.problem_from_case(_case(N), precision=0, restart=5, mg_fused=mg_fused)
    try:
        ms, by = g.time_kernel(3, 1)
        assert ms > 0 and (by > 6 * 8 * g.n_u) == stored and by >= 6 * 8 * g.n_u
    finally:
        g.close()
