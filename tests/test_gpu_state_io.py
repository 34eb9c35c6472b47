"""set_state / get_state: the values come back bit for bit, walls hold the wall
data, and the scratch they cross through fits the smallest grid and restart."""
import numpy as np
import pytest

import fsi_inputs as fi

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
@pytest.mark.parametrize("N", [2, 6, 24, 56])
def test_state_round_trip(N, precision):
    from paper_2301_10041_gb300 import fsi
    xy, tris = fi.ring_disk_mesh(1, 0.2, (0.5, 0.5))
    case = fi.FsiCase(N=N, rho_f=1.0, nu=1.0, kappa=1.0, dt=1e-2, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 3, lid_u=1.0), X0=xy.copy())
    g = fsi.problem_from_case(case, precision=precision, restart=1)
    try:
        u, p, X, lam = g.get_state()
        assert np.array_equal(u, case.u0) and np.array_equal(X, xy)
        assert not p.any() and not lam.any()
        rng = np.random.default_rng(N)
        u1, X1 = rng.standard_normal(case.u0.shape), rng.uniform(0.3, 0.7, xy.shape)
        g.set_state(u=u1)
        n1 = 2 * N + 1
        ix, iy = np.arange(n1 * n1) % n1, np.arange(n1 * n1) // n1
        inner = (ix > 0) & (iy > 0) & (ix < n1 - 1) & (iy < n1 - 1)
        want = fi.wall_velocity(N, 1.0)
        want[inner] = u1[inner]
        u, p, X, lam = g.get_state()
        assert np.array_equal(u, want) and np.array_equal(X, xy)
        g.set_state(X=X1)
        u, p, X, lam = g.get_state()
        assert np.array_equal(u, want) and np.array_equal(X, X1)
    finally:
        g.close()
