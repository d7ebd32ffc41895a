"""Gradients of the mixed element kernels on meshes padded beyond one 16-row tile (n_b 18 and 24): the
padding rows of the one-tile elements have no accumulator in a tile.  The full Frechet kernel, whose
gradient term visits every row of the padded layout, against the oracle (1e-8, the path's gradient
tolerance), checkpointed bit for bit; an adjoint session's column against the same shot alone (1e-12)."""

import numpy as np
import pytest

from oracle import uneven
from sbfwi_inputs import boundary_nodes, min_spacing, nearest_node, quadtree_mesh, ricker

pytestmark = pytest.mark.gpu

GRAD_TOL = 1e-8


def _mesh(n_b):
    if n_b == 18:                    # corner cells with hanging vertices on two sides
        m = quadtree_mesh(4, 1, lambda x0, y0, x1, y1, lvl: x0 < 0.25 or y0 < 0.25, 3)
    else:                            # a cell with four finer neighbours
        m = quadtree_mesh(3, 1, lambda x0, y0, x1, y1, lvl: not (1 / 3 <= x0 < 0.5 and 1 / 3 <= y0 < 0.5), 3)
    assert m.n_b.max() == n_b and (m.n_b <= 16).any()
    return m


def _problem(m, shots, K=30):
    rho = 0.8 + 0.4 * np.random.default_rng(shots).random((15, 15))
    s = min_spacing(m)
    dt, f0 = 0.5 * s, 1.0 / (10 * s)
    top = boundary_nodes(m, "top")
    src = np.array([nearest_node(m, top, ((k + 0.5) / shots, 1.0)) for k in range(shots)])
    wav = np.stack([(1 + 0.2 * k) * ricker(f0, dt, K, t0=1.2 / f0) for k in range(shots)])
    return rho, dt, src, wav, boundary_nodes(m, "bottom")[::2]


@pytest.mark.parametrize("n_b,shots", [(18, 8), (18, 3), (18, 2), (24, 8), (24, 5)])
def test_full_kernel(lib, n_b, shots):
    m = _mesh(n_b)
    rho, dt, src, wav, rec = _problem(m, shots)
    om = uneven.build_model(m, 5, 1.0, rho, dt)
    to, store, _, su = uneven.forward(om, src, wav, rec, keep_u=True)
    go = uneven.gradient_to_grid(om, uneven.adjoint_gradient(om, store, -to, rec, store_u=su), 15, 15)
    md = lib.Model(lib.Mesh.from_inputs(m, 5), 1.0, rho, dt)
    lib.set_schedule(md, lib.ELEMENT_MIXED)
    lib.set_kernel_terms(md, lib.TERMS_FULL)
    g = []
    for ckpt in (0, 7):
        tr, st = lib.forward(md, src, wav, rec, ckpt_every=ckpt)
        g.append(lib.adjoint_gradient(md, st, -tr))
    assert np.linalg.norm(g[0] - go) <= GRAD_TOL * np.linalg.norm(go)
    assert np.array_equal(g[0], g[1])


@pytest.mark.parametrize("n_b", [18, 24])
def test_adjoint_session(lib, n_b):
    import torch
    m = _mesh(n_b)
    rho, dt, src, wav, rec = _problem(m, 4)
    md = lib.Model(lib.Mesh.from_inputs(m, 5), 1.0, rho, dt)
    lib.set_schedule(md, lib.ELEMENT_MIXED)
    fwd = lib.Session(md, lib.SESSION_FORWARD, 4, rec, window=8)
    adj = lib.Session(md, lib.SESSION_ADJOINT, 4, rec, window=8)
    K = wav.shape[1]
    fields = [torch.zeros((K, fwd.field_stride), dtype=torch.float64, device="cuda") for _ in src]
    for k, f in enumerate(fields):
        fwd.admit(k, wav[k], int(src[k]), field=f)
    while len(fwd.step()) < len(src):
        pass
    traces = [fwd.collect(k) for k in range(len(src))]
    for k, f in enumerate(fields):
        adj.admit(k, -traces[k], field=f)
    while len(adj.step()) < len(src):
        pass
    for k in range(len(src)):
        tr, st = lib.forward(md, src[k:k + 1], wav[k:k + 1], rec)
        solo = lib.adjoint_gradient(md, st, -tr)
        assert np.abs(adj.collect(k).cpu().numpy() - solo).max() <= 1e-12 * np.abs(solo).max()


@pytest.mark.parametrize("first,then", [("MIXED", "TENSOR"), ("TENSOR", "MIXED")])
def test_session_goes_on_with_its_kernels(lib, first, then):
    """A session's operator digits outlive a later call on the model that takes the other kernels' digits."""
    m = _mesh(24)
    rho, dt, src, wav, rec = _problem(m, 4)
    md = lib.Model(lib.Mesh.from_inputs(m, 5), 1.0, rho, dt)
    lib.set_schedule(md, getattr(lib, "ELEMENT_" + first))
    solo = lib.forward(md, src, wav, rec, keep=False)[0]
    ses = lib.Session(md, lib.SESSION_FORWARD, 4, rec, window=8)
    lib.set_schedule(md, getattr(lib, "ELEMENT_" + then))
    for k in range(4):
        ses.admit(k, wav[k], int(src[k]))
    done = []
    while len(done) < 4:
        other = lib.forward(md, src, wav, rec, keep=False)[0]
        assert np.linalg.norm(other - solo) <= 1e-12 * np.linalg.norm(solo)       # the kernels' agreement
        done = ses.step()
    for k in range(4):
        assert np.abs(ses.collect(k).cpu().numpy() - solo[k]).max() <= 1e-13 * np.abs(solo).max()
