"""The exact adjoint's nodal products at the edges of their sizes: orders 1 to 7, one shot and odd
numbers of shots, the fewest radial points, against reverse-mode differentiation of the uncondensed
time loop (relative L2 1e-8, as for the path's gradients)."""

import numpy as np
import pytest

from oracle import fwi, modex, sbfem
from sbfwi_inputs import boundary_nodes, ricker, structured_mesh

pytestmark = pytest.mark.gpu

GRAD_TOL = 1e-8


@pytest.fixture(scope="module")
def lib():
    from paper_2501_06748_gb300 import sbfwi
    return sbfwi


@pytest.mark.parametrize("nx,ny,p,n_r,shots", [(1, 1, 1, 3, 1), (3, 2, 1, 4, 7), (2, 2, 4, 9, 3), (2, 1, 5, 4, 1), (1, 2, 7, 3, 2)])
def test_against_the_oracle(lib, nx, ny, p, n_r, shots):
    mesh = structured_mesh(nx, ny, p)
    pts, _ = fwi.nodal_points(mesh, sbfem.elements_from_mesh(mesh), sbfem.radial_grid(n_r - 1, 1e-3, np.float64))
    rng = np.random.default_rng(p)
    rho = 1.0 + 0.3 * rng.random(pts.shape[0])
    s = 1.0 / (max(nx, ny) * p)
    K, dt = 40, 0.4 * s
    src = rng.permutation(mesh.n_nodes)[:shots]
    rec = np.unique(boundary_nodes(mesh, "bottom"))
    wav = np.stack([(1 + 0.2 * k) * ricker(1 / (6 * s), dt, K) for k in range(shots)])
    obs = 0.01 * rng.standard_normal((shots, len(rec), K))
    md = lib.Model(lib.Mesh.from_inputs(mesh, n_r), 1.0, rho, dt, rho_kind=lib.RHO_NODAL)
    lib.set_gradient_mode(md, lib.GRAD_EXACT)
    tr, st = lib.forward(md, src, wav, rec)
    _, res = lib.misfit(tr, obs, dt)
    g = lib.adjoint_gradient(md, st, res, mode=lib.GRAD_EXACT)
    go = modex.misfit_and_gradient(mesh, n_r, 1.0, rho, dt, src, wav, rec, obs)[1]
    assert np.linalg.norm(g - go) <= GRAD_TOL * np.linalg.norm(go)
