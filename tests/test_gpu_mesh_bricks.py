"""The mesh resolver's bricks: every size of them gives the same field, lists
that overflow change nothing, and a coarse grid is not dearer than a fine one."""
import time

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


def shapes(n, lo, hi, size, seed):
    """n boxes and spheres with centres in [lo, hi] and sizes up to `size`."""
    rng = np.random.default_rng(seed)
    tris, objs, at = [], [], 0
    for q in range(n):
        c, r = rng.uniform(lo, hi), rng.uniform(0.2 * size, 0.5 * size)
        t = layouts.icosphere_mesh(*c, r, levels=1) if q % 3 == 0 else layouts.box_mesh(c[0] - r, c[0] + r, c[1] - r, c[1] + r,
                                                                                       c[2] - r, c[2] + r)
        tris.append(t)
        objs.append((at, len(t), float(rng.choice([0.0, 0.3, 0.7]))))
        at += len(t)
    return np.concatenate(tris), objs


SMALL = (20, 18, 8)
# 1, 2, 4, 8, 16 and 32 cells to a warp
SIZES = [SMALL, (37, 29, 13), (48, 40, 16), (64, 56, 20), (96, 64, 24), (128, 96, 32)]


@pytest.fixture(scope="module")
def scene():
    tris, objs = shapes(25, (4.0, 4.0, 1.0), (34.0, 30.0, 12.0), 6.0, 5)
    return tris, objs, mesh.mesh_porosity(*SMALL, 2.0, tris, objs, sub=3)


@pytest.mark.parametrize("dims", SIZES)
def test_every_brick_gives_the_same_field(dims, scene):
    tris, objs, ref = scene
    assert (ref < 1).any()
    phi = uf.Grid(*dims, h=2.0, precision="f64").mesh_to_phi(tris, objs, sub=3, set_porosity=False)
    np.testing.assert_array_equal(phi[:SMALL[2], :SMALL[1], :SMALL[0]], ref)
    if dims != SMALL:   # (the objects end before 38 m, 34 m and 16 m)
        assert (phi[:, :, 20:] == 1).all() and (phi[:, 18:, :] == 1).all() and (phi[8:] == 1).all()


# all objects in one brick: within a cell's list, past it, at the brick's list, past it (the cells look through all)
@pytest.mark.parametrize("n", [64, 65, 1024, 1025])
@pytest.mark.parametrize("dims", [(4, 3, 2), (128, 96, 32)])
def test_crowded_cells(dims, n):
    tris, objs = shapes(n, (2.5, 2.5, 1.0), (3.5, 3.5, 1.5), 1.2, n)   # around one cell of 2 m
    ref = mesh.mesh_porosity(4, 3, 2, 2.0, tris, objs, sub=2)
    phi = uf.Grid(*dims, h=2.0, precision="f64").mesh_to_phi(tris, objs, sub=2, set_porosity=False)
    np.testing.assert_array_equal(phi[:2, :3, :4], ref)


def test_many_objects_to_a_brick_few_to_a_cell():
    tris, objs = shapes(1500, (1.0, 1.0, 1.0), (23.0, 19.0, 11.0), 0.8, 3)
    ref = mesh.mesh_porosity(12, 10, 6, 2.0, tris, objs, sub=2)
    for dims in ((12, 10, 6), (128, 96, 32)):
        phi = uf.Grid(*dims, h=2.0, precision="f64").mesh_to_phi(tris, objs, sub=2, set_porosity=False)
        np.testing.assert_array_equal(phi[:6, :10, :12], ref)


def test_a_coarse_grid_is_not_dearer_than_a_fine_one():
    """300 trees on 12 x 12 x 4 cells of 25 m and on 150 x 150 x 24 of 2 m.  (With one brick size the coarse one took
    10 times as long as the fine one; it has a thousandth of the cells.)"""
    tris, objs = shapes(300, (15.0, 15.0, 2.0), (285.0, 285.0, 24.0), 12.0, 0)

    def ms(dims, h):
        g = uf.Grid(*dims, h=h)
        out = torch.empty(g.shapes["phi"], device="cuda")
        best = 1e9
        for _ in range(6):
            torch.cuda.synchronize()
            t = time.perf_counter()
            g.mesh_to_phi(tris, objs, 4, out=out)
            torch.cuda.synchronize()
            best = min(best, time.perf_counter() - t)
        return best * 1e3
    assert ms((12, 12, 4), 25.0) < 2 * ms((150, 150, 24), 2.0)
