"""The element set-up's eliminations at the edges of their sizes: fewer matrix entries than threads,
odd numbers of boundary nodes, orders whose pivots exchange rows (most steps at p = 7), working
matrices in shared and in global memory, 2-D and 3-D, against the oracle at the path's tolerance
for traces (1e-10)."""

import numpy as np
import pytest

from oracle import fwi, uneven
from sbfwi_inputs import structured_mesh, quadtree_mesh, ricker
from sbfwi_inputs.mesh3d import structured_mesh3d

pytestmark = pytest.mark.gpu

TRACE_TOL = 1e-10


def _compare(lib, mesh, n_r, spacing, extents, build, oracle):
    rng = np.random.default_rng(11)
    rho = 0.05 + 2.0 * rng.random((9,) * len(extents))
    dt, K = 0.4 * spacing, 40
    src = rng.permutation(mesh.n_nodes)[:2]
    rec = np.unique(rng.permutation(mesh.n_nodes)[:9])
    wav = np.stack([ricker(1.0 / (6 * spacing), dt, K), -0.5 * ricker(1.0 / (8 * spacing), dt, K)])
    md = lib.Model(lib.Mesh.from_inputs(mesh, n_r), 1.0, rho, dt, **extents)
    tr, _ = lib.forward(md, src, wav, rec, keep=False)
    to = oracle.forward(build(mesh, n_r, 1.0, rho, dt), src, wav, rec, keep=False)[0]
    assert np.abs(to).max() > 0
    assert np.linalg.norm(tr - to) <= TRACE_TOL * np.linalg.norm(to)


@pytest.fixture(scope="module")
def lib():
    from paper_2501_06748_gb300 import sbfwi
    return sbfwi


@pytest.mark.parametrize("p,n_r", [(1, 3), (5, 4), (6, 5), (7, 4)])
def test_squares(lib, p, n_r):
    _compare(lib, structured_mesh(3, 2, p), n_r, 1.0 / (3 * p), dict(lx=1.0, ly=1.0), fwi.build_model, fwi)


@pytest.mark.parametrize("p", [1, 3])
def test_quadtree(lib, p):
    mesh = quadtree_mesh(4, 1, lambda x0, y0, x1, y1, lvl: x0 < 0.5 and y0 < 0.5, p)
    _compare(lib, mesh, 4, 1.0 / (8 * p), dict(lx=1.0, ly=1.0), uneven.build_model, uneven)


@pytest.mark.parametrize("p", [1, 2])
def test_cubes(lib, p):
    _compare(lib, structured_mesh3d(2, 1, 2, p, lx=1.0, ly=1.0, lz=1.0), 4, 1.0 / (2 * p),
             dict(lx=1.0, ly=1.0, lz=1.0), fwi.build_model3d, fwi)
