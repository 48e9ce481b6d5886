"""GenEO eigenvalues with more copies than the eigensolver's blocks have columns
(eight).  Where Xi is one number c on the whole subdomain, B = c^2 A and every
eigenvalue of A p = lambda B p is 1 / c^2: one subdomain has c = 1, two that
coincide c = 1/2.  The kept ones must all be that value, and the coarse columns
that come with them independent (as many DOFs as columns and more here), also
where the basis comes to hold the whole space of the subdomain (54 DOFs).

Tolerance: residuals below 1e-6 mu leave the Ritz values to 1e-12; the matrices'
own rounding adds eps times their condition (1e4 at most here), so 1e-9 relative.
"""
import numpy as np
import pytest

from paper_1707_04228_gb300 import inputs

pytestmark = pytest.mark.gpu


def block(nx, ny, nz):
    lam = inputs.flat_plate_c0()
    lam.sv, lam.lv = np.linspace(0.0, nx, nx + 1), np.linspace(0.0, ny, ny + 1)
    lam.layer_nel, lam.layer_thick, lam.layer_mat, lam.layer_angle_deg = [nz], [float(nz)], [1], [0.0]
    lam.dir_dof, lam.dir_val = inputs.clamp_face(lam, inputs.FACE_SM)
    return lam


@pytest.mark.parametrize("n,px,nev,value", [
    ((1, 1, 1), 1, 9, 1.0), ((1, 1, 1), 1, 28, 1.0), ((3, 2, 1), 1, 8, 1.0), ((3, 2, 1), 1, 9, 1.0),
    ((4, 2, 2), 1, 12, 1.0), ((4, 2, 2), 1, 28, 1.0), ((2, 1, 1), 2, 9, 4.0), ((2, 1, 1), 2, 20, 4.0),
])
def test_every_copy_is_found(gl_lib, cuda_ok, n, px, nev, value):
    from paper_1707_04228_gb300 import lib
    s = lib.Solver.from_laminate(block(*n), px=px, py=1, pz=1, nev=nev)
    ev = s.geneo_eigenvalues()
    _, info = s.solve()
    s.close()
    assert ev.size == px * nev and np.all(np.abs(ev - value) <= 1e-9 * value)
    assert info["n_coarse_dropped"] == 0
