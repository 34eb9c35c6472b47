"""The coarsest grid's mirror classes on the largest coarsest grids that the
parameters allow, 24 and 32 cells: FP32 classes (from 1500 unknowns on) of the
velocity and the pressure, and FP64 class sums above 48 KB of shared memory.  Such a
grid is its own coarsest one, so the block-diagonal preconditioner's parts are direct
solves: u = A_f^-1 v_u against the oracle's block, and
p = -(nu M_p^-1 v_p + (rho / dt) L^-1 v_p) against the pressure Laplacian that the
host setup assembles (made regular by t e e^T / |e|^2, e the constants, t its mean
diagonal; condition number below 2000).  1e-11 in FP64, 1e-5 in FP32, as the smaller
grids' test."""
import os
import shutil
import subprocess

import numpy as np
import pytest
import scipy.linalg as sla
import scipy.sparse as sp
import scipy.sparse.linalg as spl

import fsi_inputs as fi
from gpu_helpers import rel
from oracle import fsi_oracle as fo

pytestmark = pytest.mark.gpu

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2301_10041_gb300", "csrc")

DUMP = r"""
#include <cstdio>
#include <cstdlib>
#include "fsi_internal.h"
int main(int argc, char** argv) {
  fsi::SetupParams sp{};
  sp.N = std::atoi(argv[1]);
  sp.rho = sp.nu = sp.kappa = sp.dt = 1.0;
  sp.npe = 3;
  sp.coarse_max = sp.coarse_max_p = sp.N;
  const double xy[6] = {0.4, 0.4, 0.6, 0.4, 0.5, 0.6};
  const int tri[3] = {0, 1, 2};
  fsi::HostSetup hs;
  fsi::build_setup(sp, 3, 1, xy, tri, hs);
  std::fwrite(hs.coarseL.data(), sizeof(double), hs.coarseL.size(), stdout);
}
"""


def _laplacian(tmp_path, N):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no C++ compiler")
    src, exe = tmp_path / "dump.cpp", str(tmp_path / "dump")
    src.write_text(DUMP)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), os.path.join(CSRC, "fsi_setup.cpp"), "-o", exe],
                   check=True)
    raw = subprocess.run([exe, str(N)], check=True, capture_output=True).stdout
    return np.frombuffer(raw).reshape(3 * N * N, 3 * N * N)


@pytest.mark.parametrize("N", [24, 32])
def test_single_level_parts_are_the_direct_solves(N, tmp_path):
    from paper_2301_10041_gb300 import fsi
    xy, tris = fi.ring_disk_mesh(3, 0.2, (0.47, 0.52))
    case = fi.FsiCase(N=N, rho_f=1.3, nu=0.05, kappa=30.0, dt=0.005, lid_u=1.0, ref_xy=xy, tris=tris,
                      u0=fi.initial_velocity(N, 7, lid_u=1.0), X0=xy.copy())
    grid = fo.FluidGrid(N)
    M, K, _ = fo.assemble_fluid(grid, case.nu)
    A = (case.rho_f / case.dt * M + K).tocsr()[grid.interior_dofs][:, grid.interior_dofs]
    L = _laplacian(tmp_path, N)
    g = fsi.problem_from_case(case, precision=1, precond=0, restart=10, mg_coarse=N)
    try:
        g.assemble_step()
        rank = np.searchsorted(grid.interior_nodes, g.interior_nodes())
        q = (2 * rank[:, None] + np.arange(2)).ravel()      # library order from the oracle's
        rng = np.random.default_rng(N)
        f, b = rng.standard_normal(g.n_u), rng.standard_normal(g.n_p)
        ref_u = spl.spsolve(sp.csc_matrix(A), f)[q]
        minv = np.tile([1.0, 12.0, 12.0], N * N) * N * N
        ref_p = -(case.nu * minv * b + case.rho_f / case.dt * sla.solve(L, b, assume_a="sym"))
        for precision, tol in ((0, 1e-11), (1, 1e-5)):
            v = np.zeros(g.n)
            v[:g.n_u] = f[q]
            # the pressure part of v is zero, so the velocity part is A_f^-1 v_u alone
            assert rel(g.apply_preconditioner(v, precision=precision)[:g.n_u], ref_u) < tol
            v = np.zeros(g.n)
            v[g.n_u:g.n_u + g.n_p] = b
            assert rel(g.apply_preconditioner(v, precision=precision)[g.n_u:g.n_u + g.n_p], ref_p) < tol
    finally:
        g.close()
