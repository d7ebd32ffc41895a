"""The tensor-core element kernels on fields near the bottom of the binary64 range, in units where the two
operators of a radial point differ by more than 2^64 (c = 1e12): the time loop is linear, so wavelets scaled by
2^-k give the traces scaled by 2^-k, up to the rounding of subnormal values (1e-12, the agreement asked of the
element kernels)."""

import numpy as np
import pytest

from sbfwi_inputs import boundary_nodes, ricker, structured_mesh

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("p,shots", [(2, 1), (4, 2), (2, 3), (4, 8), (6, 3)])
def test_traces_scale_with_the_wavelets(lib, p, shots):
    mesh = structured_mesh(4, 3, p)
    c, K = 1e12, 40
    s = 1.0 / (4 * p)
    dt = 0.5 * s / c
    src = boundary_nodes(mesh, "top")[:shots]
    rec = boundary_nodes(mesh, "bottom")
    wav = np.stack([(1 + 0.3 * k) * ricker(c / (10 * s), dt, K, t0=6 * s / c) for k in range(shots)])
    md = lib.Model(lib.Mesh.from_inputs(mesh, 6), c, np.full((8, 8), 0.9), dt)
    ref = lib.forward(md, src, wav, rec, keep=False)[0]
    assert np.abs(ref).max() > 0
    for k in range(840, 921, 8):
        tr = lib.forward(md, src, np.ldexp(wav, -k), rec, keep=False)[0]
        assert np.abs(tr).max() >= 2.0 ** -1010                    # normal numbers with bits to spare
        back = np.ldexp(tr, k)
        assert np.linalg.norm(back - ref) <= 1e-12 * np.linalg.norm(ref), k
