"""FP64 products of the factorisation on the tensor cores (integer slices): the
local factor's direct solve where the trailing matrices and panels end inside,
on and just past a tile, and where the summed range takes several exact
accumulations.

One subdomain without a coarse space is the direct solve of K_ff: its residual
with the oracle's assembled matrix is of order n eps cond, below 1e-9 on these
blocks of one stiff material (n about 1e3 to 1e4, condition below 1e4); the
laminated plate (0.02 mm resin layers: entries over many orders of magnitude in
a row) is held to the same 1e-9 as in test_gpu_tensor_core.py.
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


def plate():
    lam = inputs.flat_plate_c0()
    lam.sv, lam.lv = np.linspace(0.0, 20.0, 7), np.linspace(0.0, 20.0, 6)
    lam.dir_dof, lam.dir_val = inputs.clamp_face(lam, inputs.FACE_SM)
    return lam


@pytest.mark.parametrize("n", [(1, 1, 1), (3, 2, 1), (12, 2, 2), (5, 5, 5), (8, 7, 3), "plate"])
def test_direct_solve_residual(gl_lib, cuda_ok, n):
    from paper_1707_04228_gb300 import lib
    lam = plate() if n == "plate" else block(*n)
    sysm = fem.System(fem.Mesh(lam))
    r = inputs.random_vector(sysm.mesh.n_dof, 67)
    r[sysm.is_dir] = 0.0
    s = lib.Solver.from_laminate(lam, px=1, py=1, pz=1, nev=0)
    z = s.apply_prec(r)
    s.close()
    assert np.linalg.norm(sysm.Kff @ z[sysm.free] - r[sysm.free]) <= 1e-9 * np.linalg.norm(r)
