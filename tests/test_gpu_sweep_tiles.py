"""Sweeps with the local factors at the edges of their tiles: panels with fewer
rows and columns than one tile, with a remainder, with several tiles and with
every tile split along the summed dimension (one subdomain leaves few fronts).

One subdomain without a coarse space is the direct solve of K_ff, compared
with the oracle's: 1e-8 in FP64 (as in test_gpu_parity.py).  An FP32 factor
leaves a residual of order eps_32 x cond, below 1e-2 on these cubes of one
stiff material (condition below 1e4).
"""
import numpy as np
import pytest

from oracle import fem
from paper_1707_04228_gb300 import inputs

pytestmark = pytest.mark.gpu


def block(nx, ny, nz):
    lam = inputs.flat_plate_c0()
    lam.sv, lam.lv = np.linspace(0.0, nx, nx + 1), np.linspace(0.0, ny, ny + 1)
    lam.layer_nel, lam.layer_thick, lam.layer_mat, lam.layer_angle_deg = [nz], [float(nz)], [1], [0.0]
    lam.dir_dof, lam.dir_val = inputs.clamp_face(lam, inputs.FACE_SM)
    return lam


@pytest.mark.parametrize("n", [(1, 1, 1), (2, 1, 1), (1, 3, 2), (3, 3, 3), (9, 2, 5), (6, 6, 4)])
def test_one_subdomain_direct_solve(gl_lib, cuda_ok, n):
    from paper_1707_04228_gb300 import lib
    lam = block(*n)
    sysm = fem.System(fem.Mesh(lam))
    r = inputs.random_vector(sysm.mesh.n_dof, 61)
    r[sysm.is_dir] = 0.0
    for prec, tol in ((lib.GL_PREC_FP64, 1e-8), (lib.GL_PREC_MIXED, 1e-2)):
        s = lib.Solver.from_laminate(lam, px=1, py=1, pz=1, nev=0, precision=prec)
        z = s.apply_prec(r)
        s.close()
        assert np.abs(z[sysm.is_dir]).max() == 0.0
        assert np.linalg.norm(sysm.Kff @ z[sysm.free] - r[sysm.free]) <= tol * np.linalg.norm(r)
