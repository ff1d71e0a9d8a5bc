"""The mesh resolver beyond the sizes of its lists, bit for bit its oracle:
more objects than a brick lists, more undecided triangles than a cell lists,
more sample points than lanes, a mesh larger than the grid's scratch arrays."""
import numpy as np
import pytest

from oracle import mesh
from paper_2204_01117_gb300 import layouts, uf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uf.build()
    uf.load()


def many_objects(n):
    """n small boxes in one brick of cells, the last of them also out of it."""
    rng = np.random.default_rng(n)
    m = []
    for q in range(n):
        a = rng.uniform(0.5, 20.0, 3) * (1.0, 1.0, 0.5)
        b = a + rng.uniform(0.1, 3.0, 3)
        m.append(layouts.box_mesh(a[0], b[0], a[1], b[1], a[2], b[2]))
    return np.concatenate(m), [(12 * q, 12, float(rng.choice([0.0, 0.3, 0.6]))) for q in range(n)]


def small_spheres(levels):
    """A fine sphere inside one cell and one across eight."""
    a = layouts.icosphere_mesh(5.1, 4.9, 5.0, 0.7, levels=levels)
    b = layouts.icosphere_mesh(8.0, 8.0, 4.0, 1.5, levels=levels)
    return np.concatenate([a, b]), [(0, len(a), 0.25), (len(a), len(b), 0.5)]


CASES = {"64 objects": ((11, 10, 6), many_objects(64), 4),
         "65 objects": ((11, 10, 6), many_objects(65), 4),
         "200 objects": ((11, 10, 6), many_objects(200), 3),
         "320 triangles in a cell": ((9, 8, 5), small_spheres(2), 5),
         "larger than the scratch": ((6, 5, 4), small_spheres(3), 2),
         "sub = 16": ((4, 3, 2), (layouts.icosphere_mesh(4.0, 3.0, 2.0, 2.6, levels=0), [(0, 20, 0.4)]), 16),
         "sub = 1": ((9, 9, 5), (layouts.icosphere_mesh(9.0, 9.0, 2.0, 5.0, levels=1), [(0, 80, 0.0)]), 1)}


@pytest.mark.parametrize("name", CASES)
def test_bit_for_bit(name):
    dims, (tris, objs), sub = CASES[name]
    ref = mesh.mesh_porosity(*dims, 2.0, tris, objs, sub=sub)
    assert (ref < 1).any()
    g = uf.Grid(*dims, h=2.0, precision="f64")
    np.testing.assert_array_equal(g.mesh_to_phi(tris, objs, sub=sub, set_porosity=False), ref)
    g.mesh_to_phi(tris, objs, sub=sub)
    np.testing.assert_array_equal(g.get_state("phi"), ref)
