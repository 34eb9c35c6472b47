"""The exact rule's table of pairs takes no memory of its own where the Krylov
basis holds it, and a problem without room for it (one basis vector, a body much
finer than the grid) forms the pairs in the rows: the same C_f.  Each entry sums
the same products of positive weights either way, so the two agree to a few units
of rounding per product (1e-13 of the largest entry)."""
import numpy as np
import pytest

import fsi_inputs as fi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,rings", [(8, 30), (4, 24)])
def test_rows_without_the_table_match(N, rings):
    from paper_2301_10041_gb300 import fsi
    xy, tris = fi.ring_disk_mesh(rings, 0.2, (0.47, 0.52))
    case = fi.FsiCase(N=N, rho_f=1.3, nu=0.05, kappa=30.0, dt=0.005, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 7, lid_u=1.0), X0=xy.copy())
    table = fsi.problem_from_case(case, coupling=1, restart=250)
    rows = fsi.problem_from_case(case, coupling=1, restart=1)
    try:
        # the routes: one launch of the assembly more with the table
        assert table.graph_kernel_counts()[0] == rows.graph_kernel_counts()[0] + 1
        got = []
        for p in (table, rows):
            p.assemble_step()
            r, c, v = p.get_coupling()
            o = np.lexsort((c, r))
            got.append((r[o], c[o], v[o]))
        assert np.array_equal(got[0][0], got[1][0]) and np.array_equal(got[0][1], got[1][1])
        assert np.abs(got[0][2] - got[1][2]).max() <= 1e-13 * np.abs(got[0][2]).max()
    finally:
        table.close()
        rows.close()
