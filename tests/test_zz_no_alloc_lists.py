"""Per-cell lists of the allocation-free binning on both sides of the length a
warp sorts (256 points), against the oracle's location."""
import pytest

import fsi_inputs as fi
from test_zz_no_alloc import _check, _run_noalloc

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("N,rings", [(1, 6), (2, 7), (3, 12), (5, 12), (8, 14), (16, 14)])
def test_lists_of_every_length(N, rings):
    torch = pytest.importorskip("torch")
    from paper_2301_10041_gb300 import fsi
    xy, tris = fi.ring_disk_mesh(rings, 0.31, (0.53, 0.47))
    case = fi.FsiCase(N=N, rho_f=1.0, nu=1.0, kappa=1.0, dt=1e-2, lid_u=0.0, ref_xy=xy, tris=tris,
                      u0=fi.wall_velocity(N, 0.0), X0=xy.copy())
    _check(case, _run_noalloc(torch, fsi, case))
