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


def overlapping_ranges(n, at):
    """n objects of n triangles each, every range one triangle further on: n^2 entries of the resolver's tables."""
    tris = np.empty((2 * n, 3, 3))
    tris[:] = np.array([(0.0, 0.0, 0.0), (1.0, 0.0, 0.0), (0.0, 1.0, 0.5)]) + at
    return tris, [(i, n, 0.0) for i in range(n)]


def test_a_mesh_whose_tables_outgrow_their_index():
    """More than 2^31 entries: 46400 objects over one range of triangles.  They lie outside the domain; a cube of 12
    triangles in front of them is what the domain holds, and must come out as it does alone."""
    far, objs = overlapping_ranges(46400, at=np.array([-100.0, -100.0, -100.0]))
    cube = layouts.box_mesh(2.5, 9.2, 3.1, 8.8, 1.3, 7.7)
    g = uf.Grid(8, 7, 6, h=2.0)
    ref = g.mesh_to_phi(cube, [(0, 12, 0.25)], sub=3, set_porosity=False)
    assert (ref < 1).any()
    tris = np.concatenate([cube, far])
    phi = g.mesh_to_phi(tris, [(0, 12, 0.25)] + [(a + 12, n, p) for a, n, p in objs], sub=3, set_porosity=False)
    np.testing.assert_array_equal(phi, ref)
