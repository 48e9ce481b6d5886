"""The GenEO eigensolver where its basis fills and is restarted from its leading
Ritz vectors (64 columns up to nev = 12, 96 above): a flat plate whose kept
eigenvalues lie close together, against the oracle's dense LAPACK eigenvalues.

Tolerance 1e-7 of the largest kept one, as in test_gpu_geneo.py: the 0.02 mm resin
layers leave the matrices themselves good to about 1e-9.
"""
import re

import numpy as np
import pytest

from oracle import fem, geneo
from paper_1707_04228_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def case():
    lam = inputs.flat_plate_c0()
    lam.sv, lam.lv = np.linspace(0.0, 50.0, 4), np.linspace(0.0, 50.0, 3)
    lam.dir_dof, lam.dir_val = inputs.clamp_face(lam, inputs.FACE_SM)
    lam.px, lam.py, lam.pz = 2, 1, 1
    dec = geneo.Decomposition(fem.System(fem.Mesh(lam)), 2, 1, 1, 1)
    return lam, np.array([geneo.geneo_eigs(dec.neumann_matrix(s), s.xi, 20, method="dense")[0] for s in dec.subs])


@pytest.mark.parametrize("nev,columns", [(12, 64), (20, 96)])
def test_restart(gl_lib, cuda_ok, case, monkeypatch, capfd, nev, columns):
    from paper_1707_04228_gb300 import lib
    lam, ref = case
    monkeypatch.setenv("GL_VERBOSE", "1")
    s = lib.Solver.from_laminate(lam, nev=nev)
    monkeypatch.delenv("GL_VERBOSE")
    ev = s.geneo_eigenvalues().reshape(2, nev)
    s.close()
    steps = int(re.search(r"(\d+) block steps, basis", capfd.readouterr().err).group(1))
    assert 8 * steps > columns + 8          # more blocks than the basis holds
    scale = np.abs(ref[:, :nev]).max(axis=1, keepdims=True)
    assert np.all(np.abs(ev - ref[:, :nev]) <= 1e-7 * scale)
