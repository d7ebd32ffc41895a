"""The tensor-core element kernels at the edges of their shapes: one or two shots (a value per
lane) against the 8-shot kernel bit for bit, state in whole tiles or rows, few or many elements
per SM, one and two row tiles, against the FP64 kernel (1e-12 over a few steps)."""

import numpy as np
import pytest

from sbfwi_inputs.mesh import structured_mesh
from sbfwi_inputs.wavelet import ricker

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def lib():
    from paper_2501_06748_gb300 import sbfwi
    return sbfwi


def _problem(nx, ny, p, shots, K, scale=1.0):
    mesh = structured_mesh(nx, ny, p)
    rng = np.random.default_rng(nx * 100 + ny * 10 + p)
    rho = 1.0 + 0.5 * rng.random((10, 10))
    s = 1.0 / (max(nx, ny) * p)
    src = rng.integers(0, mesh.n_nodes, shots)
    rec = rng.permutation(mesh.n_nodes)[:5]
    wav = np.stack([scale * (1 + 0.3 * k) * ricker(0.2 / s, 0.5 * s, K) for k in range(shots)])
    return mesh, rho, 0.5 * s, src, rec, wav


@pytest.mark.parametrize("nx,ny,p,n_r", [(1, 1, 1, 3), (4, 3, 2, 6), (5, 4, 3, 7), (3, 3, 4, 9), (47, 43, 1, 4)])
@pytest.mark.parametrize("scale", [1.0, 1e-300])
def test_few_shots_match_the_batch_bit_for_bit(lib, nx, ny, p, n_r, scale):
    mesh, rho, dt, src, rec, wav = _problem(nx, ny, p, 3, 30, scale)
    md = lib.Model(lib.Mesh.from_inputs(mesh, n_r), 1.0, rho, dt)
    rec = rec[:min(len(rec), mesh.n_nodes)]
    t3, s3 = lib.forward(md, src, wav, rec)
    g3 = lib.adjoint_gradient(md, s3, -t3)
    t2, s2 = lib.forward(md, src[:2], wav[:2], rec)
    t1, s1 = lib.forward(md, src[2:], wav[2:], rec)
    assert np.array_equal(t3[:2], t2) and np.array_equal(t3[2:], t1)
    g = lib.adjoint_gradient(md, s2, -t2) + lib.adjoint_gradient(md, s1, -t1)
    # the shots' sum is formed in two parts
    assert np.abs(g - g3).max() <= 1e-14 * np.abs(g3).max() + 1e-320


@pytest.mark.parametrize("nx,ny,p,n_r,shots", [
    (5, 4, 4, 5, 8),       # whole tiles, few elements
    (5, 4, 3, 5, 5),       # whole tiles with padded rows and shots
    (5, 4, 1, 5, 3),       # rows (n_b 4)
    (50, 44, 2, 4, 7),     # rows, many elements
    (48, 46, 4, 3, 8),     # whole tiles, many elements
    (4, 3, 6, 5, 8),       # two row tiles, whole tiles
    (4, 3, 7, 5, 1),       # two row tiles, rows
])
def test_against_the_fp64_kernel(lib, nx, ny, p, n_r, shots):
    mesh, rho, dt, src, rec, wav = _problem(nx, ny, p, shots, 12)
    md = lib.Model(lib.Mesh.from_inputs(mesh, n_r), 1.0, rho, dt)
    out = []
    for element in (lib.ELEMENT_AUTO, lib.ELEMENT_FP64):
        lib.set_schedule(md, element, lib.SOLVE_AUTO)
        tr, st = lib.forward(md, src, wav, rec)
        g = lib.adjoint_gradient(md, st, -tr)
        tc, sc = lib.forward(md, src, wav, rec, ckpt_every=5)
        assert np.array_equal(tc, tr) and np.array_equal(lib.adjoint_gradient(md, sc, -tr), g)
        out.append((tr, g))
    for a, b in zip(*out):
        assert np.linalg.norm(a - b) <= 1e-12 * np.linalg.norm(b)
