"""Device memory of a problem, counted on the host (no GPU needed): for each
configuration the bytes are those that the form with every matrix stored takes
(all levels' sparse matrices, full coarsest inverses, no solid patches, no table
of coupling pairs).  The forms that replace it stay within them, so a budget that
admits the stored form admits these: by the counts alone (fsi_footprint_bytes)
and for the mesh itself (fsi_create_problem_budget).  The numbers: the stored form's
own counts, the mesh's to 256 bytes."""
import pytest

import fsi_inputs as fi

# N, rings of the disk, options: bytes by the counts, bytes for the mesh
COARSE = [   # the coarsest inverses
    (16, 3, dict(precision=0, restart=60), 39375616, 39337613),
    (16, 9, dict(precision=1, restart=60), 58466560, 58195798),
    (16, 9, dict(precision=1, restart=1), 55732736, 55462090),
    (16, 9, dict(precision=1, restart=60, mg_fused=-1, mg_cluster=-1), 58466560, 58195798),
    (24, 9, dict(precision=1, restart=60), 34382592, 33324399),
    (64, 9, dict(precision=1, restart=60), 157438720, 150683684),
    (64, 9, dict(precision=0, restart=60, mg_coarse=32), 673263104, 666547493),
]
PAIRS = [    # the exact rule's table of pairs
    (128, 50, dict(precision=1, restart=60, mg_fused=-1, coupling=1), 735133952, None),
    (16, 30, dict(precision=1, restart=60, coupling=1), 76600320, 73876072),
]
SOLID = [    # the patches of the mass solves
    (4, 30, dict(precision=1, restart=1, mg_fused=-1, mg_cluster=-1), 11008000, 9809207),
    (2, 9, dict(precision=0, restart=1, solid_law=1, gamma=1.0, eta=1.0), 1151488, 1004318),
    (24, 9, dict(precision=1, restart=60, mg_fused=-1), 36127488, 35069202),
    (64, 9, dict(precision=1, restart=1, mg_fused=-1, mg_cluster=-1, solid_law=1, gamma=1.0, eta=1.0), 124329472, 117506489),
    (6, 30, dict(precision=1, restart=60, coupling=1), 20155648, 18956814),
]


def _library():
    from paper_2301_10041_gb300 import build, fsi
    try:
        fsi.load_library(build.build())
    except RuntimeError as e:   # no toolkit on this machine
        pytest.skip(str(e))
    return fsi


def _params(fsi, N, opt):
    return fsi.make_params(N, 1.0, 0.01, 10.0, 1e-3, **opt)


def _admits(fsi, prm, xy, tris, budget):
    """Whether a creation under the budget gets past it (without a GPU it then
    ends in a CUDA error)."""
    try:
        fsi.Problem(prm, xy, tris, X0=xy.copy(), budget_bytes=budget).close()
        return True
    except fsi.FsiError as e:
        assert e.code in (fsi.FSI_ERR_BUDGET, fsi.FSI_ERR_CUDA, fsi.FSI_ERR_OOM)
        return e.code != fsi.FSI_ERR_BUDGET


@pytest.mark.parametrize("N,rings,opt,counts,mesh", COARSE + PAIRS + SOLID)
def test_budgets_of_the_stored_form_still_admit(N, rings, opt, counts, mesh):
    fsi = _library()
    xy, tris = fi.ring_disk_mesh(rings, 0.2, (0.47, 0.52))
    prm = _params(fsi, N, opt)
    by_counts = fsi.footprint_bytes(prm, xy.shape[0], tris.shape[0])
    assert 0 < by_counts <= counts
    assert mesh is None or _admits(fsi, prm, xy, tris, mesh)
    assert _admits(fsi, prm, xy, tris, by_counts)       # the counts bound every mesh
    assert not _admits(fsi, prm, xy, tris, by_counts // 4)


@pytest.mark.parametrize("N,rings,opt,counts", [
    (128, 25, dict(precision=1, restart=60), 516639744),
    (128, 25, dict(precision=0, restart=60), 458216960),
])
def test_matrix_free_levels_hold_no_stored_matrices(N, rings, opt, counts):
    """Neither the operator nor the finest level keeps its velocity block (2 x 2
    values and a column per block, 16 blocks a row: one of each at least)."""
    fsi = _library()
    xy, tris = fi.ring_disk_mesh(rings, 0.2, (0.47, 0.52))
    by_counts = fsi.footprint_bytes(_params(fsi, N, opt), xy.shape[0], tris.shape[0])
    block = 4 * (4 if opt["precision"] else 8) + 4
    assert counts - by_counts >= 2 * 15 * (2 * N - 1) ** 2 * block
