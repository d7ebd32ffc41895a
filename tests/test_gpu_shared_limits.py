"""A time loop that is kept (a session) next to other calls that need less shared memory in the same kernels:
the other calls leave the kernels' limits where the session's launches need them."""

import numpy as np
import pytest

from sbfwi_inputs import boundary_nodes, ricker, structured_mesh

pytestmark = pytest.mark.gpu


def _model(lib, nx, p, n_r, element):
    m = structured_mesh(nx, nx, p)
    s = 1.0 / (nx * p)
    md = lib.Model(lib.Mesh.from_inputs(m, n_r), 1.0, 1.0 + 0.3 * np.random.default_rng(nx).random((9, 9)), 0.5 * s)
    lib.set_schedule(md, element)
    return m, md, s


@pytest.mark.parametrize("element,nx,n_r,other_nx,other_n_r,other_shots", [
    ("AUTO", 32, 3, 8, 3, 12),        # the solve's staging: 60 KB, then less with other fronts or shots
    ("AUTO", 32, 3, 20, 3, 8),
    ("AUTO", 32, 3, 10, 3, 16),
    ("FP64", 3, 41, 3, 40, 8),        # operators copied ahead: 50 KB, then 49 KB
])
def test_session_between_forwards(lib, element, nx, n_r, other_nx, other_n_r, other_shots):
    element = getattr(lib, "ELEMENT_" + element)
    m, md, s = _model(lib, nx, 4, n_r, element)
    K, rec = 24, boundary_nodes(m, "bottom")[::5]
    src = boundary_nodes(m, "top")[1:9]
    wav = np.stack([(1 + 0.1 * k) * ricker(1 / (10 * s), 0.5 * s, K, t0=8 * s) for k in range(8)])
    solo = lib.forward(md, src, wav, rec, keep=False)[0]
    m2, md2, s2 = _model(lib, other_nx, 4, other_n_r, lib.ELEMENT_AUTO if element == lib.ELEMENT_AUTO else element)
    src2 = np.resize(boundary_nodes(m2, "top"), other_shots)
    wav2 = np.stack([ricker(1 / (10 * s2), 0.5 * s2, 5, t0=2 * s2) for _ in range(other_shots)])
    ses = lib.Session(md, lib.SESSION_FORWARD, 8, rec, window=8)
    for k in range(8):
        ses.admit(k, wav[k], int(src[k]))
    done = []
    while len(done) < 8:
        lib.forward(md2, src2, wav2, boundary_nodes(m2, "bottom"), keep=False)
        done = ses.step()
    for k in range(8):
        assert np.abs(ses.collect(k).cpu().numpy() - solo[k]).max() <= 1e-13 * np.abs(solo).max()
