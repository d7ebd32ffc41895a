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


@pytest.mark.parametrize("nx,ny,p,n_r,shots", [
    (4, 3, 4, 4, 8),      # one element a block, operators copied ahead in 16-byte pieces
    (4, 3, 1, 3, 2),      # sixteen elements a block, the last block short
    (3, 2, 5, 3, 5),      # n_b 20
    (2, 2, 4, 40, 8),     # too many radial points to stage
    (40, 33, 4, 3, 3),    # more blocks of two elements than fit the SMs at once: direct
])
def test_operators_copied_ahead_or_not(lib, nx, ny, p, n_r, shots):
    """The transposed sweeps against the derivative along one direction: <g, d> and the misfit's central
    difference (truncation h^2, rounding 1e-13 / h of the misfit: 1e-5 at h = 1e-4)."""
    mesh = structured_mesh(nx, ny, p)
    rng = np.random.default_rng(nx)
    M = lib.Mesh.from_inputs(mesh, n_r)
    rho, d = 1.0 + 0.3 * rng.random(M.n_nodal), rng.standard_normal(M.n_nodal)
    s = 1.0 / (max(nx, ny) * p)
    K, dt = 25, 0.4 * s
    src = rng.permutation(mesh.n_nodes)[:shots]
    wav = np.stack([(1 + 0.2 * k) * ricker(1 / (6 * s), dt, K) for k in range(shots)])
    obs = np.zeros((shots, shots, K))

    def run(r, gradient):
        md = lib.Model(M, 1.0, r, dt, rho_kind=lib.RHO_NODAL)
        lib.set_gradient_mode(md, lib.GRAD_EXACT)
        tr, st = lib.forward(md, src, wav, np.sort(src))
        E, res = lib.misfit(tr, obs, dt)
        return E, lib.adjoint_gradient(md, st, res, mode=lib.GRAD_EXACT) if gradient else None

    h = 1e-4
    g = run(rho, True)[1]
    fd = (run(rho + h * d, False)[0] - run(rho - h * d, False)[0]) / (2 * h)
    assert abs(g @ d - fd) <= 1e-5 * abs(fd)
