"""The inverses of the global matrix's separator blocks by clusters of blocks: separators from one node to
one more than a cluster holds, clusters of 1 to 8 with slabs that do not divide evenly, against the
oracle's sparse LU (1e-10 on traces)."""

import numpy as np
import pytest

from oracle import fwi
from sbfwi_inputs import structured_mesh, ricker
from sbfwi_inputs.mesh3d import structured_mesh3d

pytestmark = pytest.mark.gpu

TRACE_TOL = 1e-10


@pytest.fixture(scope="module")
def lib():
    from paper_2501_06748_gb300 import sbfwi
    return sbfwi


@pytest.mark.parametrize("nx,ny,p", [
    (1, 1, 1),        # no separator but the whole element
    (2, 1, 1),        # separators of two nodes
    (9, 7, 2),        # 15 and 19 nodes
    (16, 12, 3),      # up to 49 nodes, clusters of 2 and 4
    (33, 30, 1),      # up to 34 nodes, many small fronts
    (30, 26, 4),      # up to 121 nodes: clusters of 8, slabs of 16 that leave the last short
])
def test_squares(lib, nx, ny, p):
    _compare(lib, structured_mesh(nx, ny, p), 1.0 / (max(nx, ny) * p), dict(lx=1.0, ly=1.0), fwi.build_model)


@pytest.mark.parametrize("m", [7, 10])
def test_cubes(lib, m):
    """Separators of up to 225 and 441 nodes (a cluster holds 440)."""
    _compare(lib, structured_mesh3d(m, m, m, 2, lx=1.0, ly=1.0, lz=1.0), 0.5 / m, dict(lx=1.0, ly=1.0, lz=1.0),
             fwi.build_model3d)


def _compare(lib, mesh, spacing, extents, build):
    rng = np.random.default_rng(5)
    rho = 0.7 + 0.6 * rng.random((9,) * len(extents))
    n_r, dt, K = 3, 0.5 * spacing, 25
    src = rng.permutation(mesh.n_nodes)[:2]
    rec = np.unique(rng.permutation(mesh.n_nodes)[:9])
    wav = np.stack([ricker(1.0 / (6 * spacing), dt, K), -0.5 * ricker(1.0 / (8 * spacing), dt, K)])
    md = lib.Model(lib.Mesh.from_inputs(mesh, n_r), 1.0, rho, dt, **extents)
    tr, _ = lib.forward(md, src, wav, rec, keep=False)
    to = fwi.forward(build(mesh, n_r, 1.0, rho, dt), src, wav, rec, keep=False)[0]
    assert np.abs(to).max() > 0
    assert np.linalg.norm(tr - to) <= TRACE_TOL * np.linalg.norm(to)
