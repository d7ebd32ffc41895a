"""The factor entries that a mesh reports are those of the solve's grouped levels, which a model keeps."""

import pytest

from sbfwi_inputs import structured_mesh


@pytest.mark.parametrize("nx,ny,p", [(1, 1, 3), (2, 2, 1), (3, 2, 2)])
def test_one_group_is_one_dense_inverse(nx, ny, p):
    from paper_2501_06748_gb300 import build
    build.build()
    from paper_2501_06748_gb300 import sbfwi
    M = sbfwi.Mesh.from_inputs(structured_mesh(nx, ny, p), 4)
    # meshes this small are eliminated in one group of levels: an inverse of all boundary nodes
    assert M.factor_entries == M.n_nodes ** 2
