"""C_f rows by the point rule where their kernel changes: windows too large for
three copies (bodies coarser than the grid), rows of several batches of 32 points
(a fan's hub), the last batch ragged, and rows at the walls under a moving lid.
Reference: the oracle's coupling matrix; 1e-13 of the largest entry, the bound of
the parity suite (some 40 products per entry)."""
import numpy as np
import pytest

import fsi_inputs as fi
from oracle import fsi_oracle as fo

pytestmark = pytest.mark.gpu


def _fan(n):
    th = 2 * np.pi * np.arange(n) / n
    xy = np.concatenate([[[0.5, 0.5]], 0.5 + 0.09 * np.stack([np.cos(th), np.sin(th)], 1)])
    return xy, np.array([(0, 1 + i, 1 + (i + 1) % n) for i in range(n)], dtype=np.int32)


CASES = {
    "coarse body": (16, lambda: fi.ring_disk_mesh(1, 0.3, (0.5, 0.5))),      # window of about 21 x 21 nodes
    "coarse body, finer grid": (20, lambda: fi.ring_disk_mesh(2, 0.4, (0.5, 0.5))),
    "fine body": (16, lambda: fi.ring_disk_mesh(14, 0.2, (0.43, 0.57))),
    "hub of 7": (24, lambda: _fan(7)),
    "hub of 40": (24, lambda: _fan(40)),
    "quads": (16, lambda: fi.annulus_mesh(2, 3, quads=True)),
    "under the lid": (16, lambda: fi.ring_disk_mesh(5, 0.07, (0.43, 0.925))),
}


@pytest.mark.parametrize("name", list(CASES))
def test_rows_match_the_oracle(name):
    from paper_2301_10041_gb300 import fsi
    N, mesh = CASES[name]
    xy, tris = mesh()
    case = fi.FsiCase(N=N, rho_f=1.0, nu=1.0, kappa=10.0, dt=1e-2, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 3, lid_u=1.0), X0=xy.copy())
    o = fo.OracleProblem(case.N, case.rho_f, case.nu, case.kappa, case.dt, case.lid_u, case.ref_xy, case.tris)
    grid = fo.FluidGrid(N)
    assemble = fo.assemble_coupling_q1 if tris.shape[1] == 4 else fo.assemble_coupling
    C = assemble(grid, xy, tris.astype(np.int64), case.X0)
    C = np.asarray((C[0] if isinstance(C, tuple) else C).todense())
    _, rhs, _ = o.system(case.u0, case.X0)
    g = fsi.problem_from_case(case, restart=10)
    try:
        g.assemble_step()
        rows, cols, vals = g.get_coupling()
        b = g.get_rhs()
        n_x = g.n_x
    finally:
        g.close()
    got = np.zeros_like(C)
    got[rows, cols] = vals
    inner = np.zeros(C.shape[1], dtype=bool)
    inner[grid.interior_nodes] = True
    assert np.max(np.abs(got[:, inner] - C[:, inner])) <= 1e-13 * np.max(np.abs(C))
    assert not got[:, ~inner].any()
    lam = b[-n_x:]          # -(1/dt) C_s X - C_D u_D: the wall columns
    assert np.linalg.norm(lam - rhs[-n_x:]) <= 1e-13 * np.linalg.norm(rhs[-n_x:])
