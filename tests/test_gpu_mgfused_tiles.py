"""The 16-node velocity tiles of the fused levels above 128 cells at every smoothing
degree (the frames grow with the degree, up to one CTA per SM by shared memory),
against the stored matrices (mg_fused = -1): the same preconditioner up to FP32
rounding, 2e-5 as at the other sizes.  160 cells leave ragged tiles, 256 none."""
import numpy as np
import pytest

import fsi_inputs as fi
from gpu_helpers import rel

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("degree", [1, 2, 3, 4])
@pytest.mark.parametrize("N", [160, 256])
def test_large_tiles_match_the_stored_levels(N, degree):
    from paper_2301_10041_gb300 import fsi
    xy, tris = fi.ring_disk_mesh(12, 0.2, (0.47, 0.52))
    case = fi.FsiCase(N=N, rho_f=1.0, nu=0.01, kappa=100.0, dt=1e-3, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 7, lid_u=1.0), X0=xy.copy())
    kw = dict(precision=1, precond=2, stokes_its=2, restart=5, mg_degree=degree)
    on = fsi.problem_from_case(case, **kw)
    off = fsi.problem_from_case(case, mg_fused=-1, **kw)
    try:
        on.assemble_step()
        off.assemble_step()
        assert on.graph_kernel_counts()[3] < off.graph_kernel_counts()[3]
        v = np.random.default_rng(3).standard_normal(on.n)
        assert rel(on.apply_preconditioner(v, precision=1), off.apply_preconditioner(v, precision=1)) < 2e-5
    finally:
        on.close()
        off.close()
