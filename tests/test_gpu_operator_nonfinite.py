"""An infinite entry of the operand reaches only the rows that hold its column:
the other rows of A x keep the bits they have with a finite entry there (the
C_f^T rows load their entries in groups, and the places past a row's end must
not read another row's operand).  The pattern is the oracle's."""
import numpy as np
import pytest

import fsi_inputs as fi
from gpu_helpers import oracle_to_gpu_perm
from oracle import fsi_oracle as fo

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,precision", [(16, 1), (32, 0), (64, 0), (64, 1)])
def test_infinite_multiplier_stays_in_its_rows(N, precision):
    from paper_2301_10041_gb300 import fsi
    xy, tris = fi.ring_disk_mesh(max(2, N // 8), 0.2, (0.47, 0.52))
    case = fi.FsiCase(N=N, rho_f=1.3, nu=0.05, kappa=30.0, dt=0.005, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 7, lid_u=1.0), X0=xy.copy())
    o = fo.OracleProblem(case.N, case.rho_f, case.nu, case.kappa, case.dt, case.lid_u, case.ref_xy, case.tris)
    K, _, _ = o.system(case.u0, case.X0)
    g = fsi.problem_from_case(case, precision=1, restart=20)
    try:
        g.assemble_step()
        q = oracle_to_gpu_perm(o, g)
        n_s = xy.shape[0]
        for node in (0, n_s // 2):                       # node 0 is the place an absent entry would read
            lam = g.n - 2 * n_s + 2 * node
            x = np.random.default_rng(3).standard_normal(g.n)
            ref = g.apply_operator(x, precision=precision)
            x[lam] = x[lam + 1] = np.inf
            y = g.apply_operator(x, precision=precision)
            touched = np.asarray((abs(K.tocsr()[q][:, q[[lam, lam + 1]]])).sum(axis=1)).ravel() != 0
            assert np.count_nonzero(touched) > 0
            # C_f and C_s act on both components alike: the other component's rows
            # hold zeros or nothing at these columns
            pair = touched.copy()
            for a in (0, g.n_u + g.n_p):
                b = g.n_u if a == 0 else g.n
                pair[a:b] = np.repeat(touched[a:b].reshape(-1, 2).any(axis=1), 2)
            assert np.array_equal(y[~pair], ref[~pair])
    finally:
        g.close()
