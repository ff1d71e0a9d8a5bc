"""Meshes and grids at the far end of what the mesh resolver takes."""
import numpy as np
import pytest

from paper_2204_01117_gb300 import layouts, uf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uf.build()
    uf.load()


# four planes to a brick: 65536 layers of bricks, and one more
@pytest.mark.parametrize("nz", [262144, 262145])
def test_more_layers_of_bricks_than_a_grid_dimension_holds(nz):
    nx, ny, h = 9, 2, 2.0
    box = layouts.box_mesh(8 * h, 9 * h, 0.0, h, (nz - 2) * h, nz * h)   # the last two cells of a column
    g = uf.Grid(nx, ny, nz, h=h)
    phi = g.mesh_to_phi(box, [(0, len(box), 0.0)], sub=2, set_porosity=False)
    ref = np.ones((nz, ny, nx), dtype=phi.dtype)
    ref[nz - 2:, 0, 8] = 0.0
    np.testing.assert_array_equal(phi, ref)
