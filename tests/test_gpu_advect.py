"""The two forms of the fused advection (displacements below one cell, and any
displacement) and its automatic block depth: bit for bit the separate
sub-step kernels, whatever the Courant number and the depth."""
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


def steps(dims, precision, deg, n=2, unfused=0, zc=0, **extra):
    nx, ny, nz = dims
    sc = layouts.urban_block(nx, ny, nz, h=2.0, n_boxes=2, n_trees=2, seed=1, footprint=(6.0, 10.0), height=(3.0, 8.0),
                             wind_dir_deg=deg)
    g = uf.Grid(nx, ny, nz, precision=precision, **{**sc.params(), **extra})
    g.set_tuning(unfused=unfused, advect_zc=zc)
    g.set_porosity(sc.phi.astype(g.np_dtype))
    g.init_state()
    g.run(n)
    return g.state()


# every point on a lattice end (2 x 2), one cell in z, a block without ends (100 x 40), the ends inside a tile
@pytest.mark.parametrize("dims, deg", [((24, 24, 1), 90.0), ((33, 17, 2), 200.0), ((100, 42, 7), 45.0), ((34, 26, 19), 300.0)])
@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("cfl", [0.5, 0.999, 1.0, 2.5])
def test_equals_sub_step_kernels(dims, deg, precision, cfl):
    a = steps(dims, precision, deg, cfl=cfl)
    b = steps(dims, precision, deg, unfused=uf.UNFUSED_ADVECT, cfl=cfl)
    for n in a:
        np.testing.assert_array_equal(a[n], b[n], err_msg=n)


@pytest.mark.parametrize("zc", [1, 3, 16, 64])
def test_depth_does_not_matter(zc):
    a, b = steps((70, 30, 21), "f32", 20.0), steps((70, 30, 21), "f32", 20.0, zc=zc)
    for n in a:
        np.testing.assert_array_equal(a[n], b[n], err_msg=n)
