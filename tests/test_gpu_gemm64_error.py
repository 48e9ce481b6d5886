"""FP64 accuracy of the factorisation's products on the tensor cores (integer
digits), and numbers that are none.

One subdomain without a coarse space is the direct solve of K_ff.  Its residual is
held to five times that of SciPy's sparse LU (FP64 throughout) on the same system
and right-hand sides: both are backward stable up to the same powers of n, and a
factor of five covers the different orderings, element matrices and the panels'
inverse form.  Two low digits lost of the eight would cost 2^16.  The cases end
their trailing matrices, panels and pivot blocks inside, on and past a tile, and
sum over several exact accumulations.
"""
import numpy as np
import pytest
import scipy.sparse.linalg as spla

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


@pytest.mark.parametrize("n", [(1, 1, 1), (3, 2, 1), (12, 2, 2), (5, 5, 5), (8, 7, 3), "plate", "corner"])
def test_residual_of_fp64_products(gl_lib, cuda_ok, n):
    from paper_1707_04228_gb300 import lib
    lam = plate() if n == "plate" else inputs.corner_mini() if n == "corner" else block(*n)
    sysm = fem.System(fem.Mesh(lam))
    lu = spla.splu(sysm.Kff.tocsc())
    s = lib.Solver.from_laminate(lam, px=1, py=1, pz=1, nev=0)
    ours, scipys = [], []
    for seed in (71, 72, 73):
        r = inputs.random_vector(sysm.mesh.n_dof, seed)
        r[sysm.is_dir] = 0.0
        b = r[sysm.free]
        resid = lambda x: np.linalg.norm(sysm.Kff @ x - b) / np.linalg.norm(b)
        ours.append(resid(s.apply_prec(r)[sysm.free]))
        scipys.append(resid(lu.solve(b)))
    s.close()
    assert np.linalg.norm(ours) <= 5.0 * np.linalg.norm(scipys)


@pytest.mark.parametrize("value", [np.nan, np.inf])
@pytest.mark.parametrize("where", [0, -1])
def test_not_a_number_is_reported(gl_lib, cuda_ok, value, where):
    """An element whose stiffness is not a number makes a pivot that is not positive, wherever it lies in the
    tiles: the set-up reports it, and the library serves the next one."""
    from paper_1707_04228_gb300 import lib
    lam = block(5, 3, 3)
    lam.materials = [m for m in lam.materials if m["kind"] == "ortho"] + [dict(inputs.RESIN_T1)]
    lam.layer_mat = [0]
    theta = np.zeros(45)
    theta[where] = value
    lam.theta = theta
    with pytest.raises(lib.GLError) as e:
        lib.Solver.from_laminate(lam, px=1, py=1, pz=1, nev=0)
    assert e.value.code == -4          # GL_ERR_NOT_SPD
    lam.theta = None
    s = lib.Solver.from_laminate(lam, px=1, py=1, pz=1, nev=0)
    _, info = s.solve()
    s.close()
    assert info["status"] == 0
