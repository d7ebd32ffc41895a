"""The per-step global solve on the grouped elimination tree: meshes whose levels fall into one,
two or more groups (one element, odd halvings, elements that eliminate nothing), every solve
schedule bit for bit the same and within the oracle's bounds, forward and adjoint."""

import numpy as np
import pytest

from oracle import fwi
from sbfwi_inputs.mesh import structured_mesh
from sbfwi_inputs.wavelet import ricker

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2501_06748_gb300 import sbfwi
    return sbfwi


def _rel(a, b):
    return np.linalg.norm(a - b) / np.linalg.norm(b)


@pytest.mark.parametrize("nx,ny,p,shots", [(1, 1, 2, 1), (2, 1, 3, 2), (3, 2, 1, 8), (7, 5, 2, 3), (13, 9, 2, 11),
                                           (20, 17, 1, 4)])
def test_grouped_levels(lib, nx, ny, p, shots):
    mesh = structured_mesh(nx, ny, p)
    n_r, K, grid = 5, 24, 12
    rng = np.random.default_rng(nx + 31 * ny)
    rho = 1.0 + 0.5 * rng.random((grid, grid))
    s = 1.0 / (max(nx, ny) * p)
    dt = 0.5 * s
    src = rng.integers(0, mesh.n_nodes, shots)
    rec = rng.permutation(mesh.n_nodes)[:min(6, mesh.n_nodes)]
    wav = np.stack([(1 + 0.1 * k) * ricker(0.2 / s, dt, K) for k in range(shots)])
    om = fwi.build_model(mesh, n_r, 1.0, rho, dt)
    to, store, _ = fwi.forward(om, src, wav, rec)
    go = fwi.gradient_to_grid(om, fwi.adjoint_gradient(om, store, -to, rec), grid, grid)
    M = lib.Mesh.from_inputs(mesh, n_r)
    md = lib.Model(M, 1.0, rho, dt)
    out = {}
    for solve in (lib.SOLVE_DATAFLOW, lib.SOLVE_BARRIER, lib.SOLVE_LEVELS):
        lib.set_schedule(md, lib.ELEMENT_AUTO, solve)
        tr, st = lib.forward(md, src, wav, rec)
        out[solve] = tr, lib.adjoint_gradient(md, st, -tr)
    tr, g = out[lib.SOLVE_DATAFLOW]
    for solve in (lib.SOLVE_BARRIER, lib.SOLVE_LEVELS):
        assert np.array_equal(out[solve][0], tr) and np.array_equal(out[solve][1], g)
    assert _rel(tr, to) <= 1e-10
    assert _rel(g, go) <= 1e-8
