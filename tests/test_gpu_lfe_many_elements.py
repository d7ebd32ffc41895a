"""The comparison method's element set-up with more elements than SMs, so that blocks share an SM and their warps
drift apart: traces and gradient against the oracle (1e-10, 1e-8) and every set-up the same bits."""

import numpy as np
import pytest

from oracle import fwi, lfe
from sbfwi_inputs import boundary_nodes, ricker, structured_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nx,ny,p", [(26, 20, 2), (14, 13, 4), (40, 31, 1)])
def test_many_elements(lib, nx, ny, p):
    m = structured_mesh(nx, ny, p)
    rng = np.random.default_rng(nx)
    rho = 0.8 + 0.4 * rng.random((17, 17))
    s = 1.0 / (max(nx, ny) * p)
    dt, K = 0.45 * s, 25
    src = boundary_nodes(m, "top")[[2, -5]]
    rec = boundary_nodes(m, "top")[::7]
    wav = np.stack([ricker(1 / (8 * s), dt, K, t0=5 * s), -0.5 * ricker(1 / (9 * s), dt, K, t0=6 * s)])
    to, Eo, go = lfe.forward_and_gradient(m, 1.0, fwi.grid_to_points(rho, m.node_xy, 1.0, 1.0), dt, src, wav, rec,
                                          np.zeros((2, rec.size, K)))
    M = lib.Mesh.from_inputs(m, 3)
    runs = []
    for _ in range(3):
        md = lib.Model(M, 1.0, rho, dt, lfe=True)
        tr, st = lib.forward(md, src, wav, rec)
        E, res = lib.misfit(tr, np.zeros_like(tr), dt)
        runs.append((tr, lib.adjoint_gradient(md, st, res)))
    tr, g = runs[0]
    assert np.abs(to).max() > 0
    assert np.linalg.norm(tr - to) <= 1e-10 * np.linalg.norm(to)
    gog = fwi.points_to_grid(go, m.node_xy, 17, 17, 1.0, 1.0)
    assert np.linalg.norm(g - gog) <= 1e-8 * np.linalg.norm(gog)
    for other in runs[1:]:
        assert np.array_equal(other[0], tr) and np.array_equal(other[1], g)
