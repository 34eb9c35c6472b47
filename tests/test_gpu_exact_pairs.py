"""C_f by the exact rule where a node's triangles take both routes: those over at
most four cells from the pair table, the wider ones formed in the rows; and
triangles with vertices on grid lines and corners.

Tolerance: an entry sums at most a few hundred products; the coordinates carry
eps / (triangle's size in the unit square) <= 1e-14 relative and each product a
few eps, so 1e-13 of the largest entry holds with room.
"""
import numpy as np
import pytest
import scipy.sparse as sp

import fsi_inputs as fi
from oracle import fsi_oracle as fo

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def fsi():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2301_10041_gb300 import build, fsi as f
    build.build()
    f.load_library()
    return f


def boxes(tris, X, N):
    """Number of fluid cells in each triangle's bounding box (last cell closed)."""
    c = np.minimum(np.floor(X * N).astype(int), N - 1)[tris]
    return np.prod(c.max(1) - c.min(1) + 1, axis=1)


def case(N, m, stretch, snap):
    xy, tris = fi.ring_disk_mesh(m, 0.3, (0.5, 0.5))
    X = (xy - 0.5) * np.array([1.0, stretch]) + 0.5
    if snap:                       # coordinates near a grid line onto it
        r = np.round(X * N)
        X = np.where(np.abs(X * N - r) < 0.15, r / N, X)
    return fi.FsiCase(N=N, rho_f=1.0, nu=0.5, kappa=20.0, dt=0.01, lid_u=0.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 3), X0=X, precond=1, rtol=1e-12)


CASES = [(24, 5, 1.0, False), (24, 6, 0.7, True), (32, 8, 1.2, False), (16, 6, 1.0, True), (40, 8, 1.0, False)]


@pytest.mark.parametrize("N,m,stretch,snap", CASES)
def test_exact_coupling_both_routes(fsi, N, m, stretch, snap):
    c = case(N, m, stretch, snap)
    g = fsi.problem_from_case(c, coupling=1)
    g.assemble_step()
    rows, cols, vals = g.get_coupling()
    g.close()
    grid = fo.FluidGrid(N)
    C = fo.assemble_coupling_exact(grid, c.ref_xy, c.tris.astype(np.int64), c.X0)
    C = C.tocsc()[:, grid.interior_nodes].tocsr()
    G = sp.coo_matrix((vals, (rows, np.searchsorted(grid.interior_nodes, cols))), shape=C.shape).tocsr()
    assert abs(G - C).max() <= 1e-13 * abs(C).max()


@pytest.mark.parametrize("N,m,stretch,snap", CASES)
def test_cases_hold_both_routes(N, m, stretch, snap):
    c = case(N, m, stretch, snap)
    b = boxes(c.tris, c.X0, N)
    assert (b <= 4).any() and (b > 4).any()
