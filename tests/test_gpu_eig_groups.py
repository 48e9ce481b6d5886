"""eig_group_bytes bounds the eigensolver's memory: a group's Krylov basis counts
beside its factors.

A row of 12 elements in 12 subdomains: with an element of overlap on either side
a subdomain has at most 7 x 3 x 3 nodes, 189 DOFs, all of them 10 x 189 + 135 + 108
(one end free, one clamped).  A factor has at most as many entries per DOF as the
subdomain has DOFs, 1,512 bytes; the basis for nev = 28 takes 2,848.  So 2,000
bytes per DOF hold all factors but not both, and 4,400 hold everything.  The
eigenvalues are the same within the eigensolver's convergence (residuals of
1e-6, so 1e-9 of the largest kept one)."""
import numpy as np
import pytest

from paper_1707_04228_gb300 import inputs

pytestmark = pytest.mark.gpu

DOFS = 10 * 189 + 135 + 108


def test_basis_counts(gl_lib, cuda_ok):
    from paper_1707_04228_gb300 import lib
    lam = inputs.flat_plate_c0()
    lam.sv, lam.lv = np.linspace(0.0, 12.0, 13), np.linspace(0.0, 1.0, 2)
    lam.layer_nel, lam.layer_thick, lam.layer_mat, lam.layer_angle_deg = [1], [1.0], [1], [0.0]
    lam.dir_dof, lam.dir_val = inputs.clamp_face(lam, inputs.FACE_SM)
    ev = []
    for bytes_per_dof, one in ((4400.0, True), (2000.0, False)):
        s = lib.Solver.from_laminate(lam, px=12, py=1, pz=1, nev=28, eig_group_bytes=bytes_per_dof * DOFS)
        assert (s.profile_read()["eig_groups"] == 1) == one
        ev.append(s.geneo_eigenvalues())
        _, info = s.solve()
        assert info["status"] == 0
        s.close()
    assert np.abs(ev[0] - ev[1]).max() <= 1e-9 * np.abs(ev[0]).max()
