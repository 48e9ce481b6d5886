"""The eigensolver's sweeps with eight vectors on the tensor cores (integer
slices): fronts below one tile, with remainders in both directions, and with
several tiles and several exact accumulations along the summed dimension.

The kept eigenvalues against the oracle's dense LAPACK eigenvalues: residuals
below 1e-6 leave the Ritz values to second order in it, so 1e-9 of each
subdomain's largest kept one; 1e-7 (as in test_gpu_geneo.py) covers LAPACK's
own error on the zero eigenvalues of floating subdomains.
"""
import numpy as np
import pytest

from oracle import fem, geneo
from paper_1707_04228_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n_arc,n_width,angles,nsub,nev", [
    (2, 1, (0,), (2, 1, 1), 2),
    (2, 1, (0, 45, 90), (2, 1, 1), 3),
    (4, 2, (0, 45, 90), (2, 1, 1), 8),
    (7, 3, (0, 45, 90), (3, 1, 1), 10),
])
def test_eigenvalues_by_front_size(gl_lib, cuda_ok, n_arc, n_width, angles, nsub, nev):
    from paper_1707_04228_gb300 import lib
    lam = inputs.corner_mini(n_arc=n_arc, n_limb=1, n_width=n_width, nel_layer=1, angles=angles, nsub=nsub, nev=nev,
                             limb_L=3.0, width=3.0)
    sysm = fem.System(fem.Mesh(lam))
    dec = geneo.Decomposition(sysm, lam.px, lam.py, lam.pz, 1)
    ref = np.array(geneo.GenEO(dec, nev, eig_method="dense").eigvals)
    s = lib.Solver.from_laminate(lam)
    ev = s.geneo_eigenvalues().reshape(len(dec.subs), nev)
    s.close()
    scale = np.abs(ref).max(axis=1, keepdims=True)
    assert np.all(np.abs(ev - ref) <= 1e-7 * np.maximum(scale, 1.0))
