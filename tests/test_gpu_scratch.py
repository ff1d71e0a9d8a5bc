"""The step's scratch arrays are lent to other calls (field transfers, the
autotuner, the mesh resolver).  What these leave there, row padding included,
must not reach a state initialised afterwards, whose first time step is the
CFL maximum over whole arrays."""
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


def use_mesh(g):
    tris, objects = layouts.mesh_city(g.desc.nx, g.desc.ny, g.desc.nz, g.desc.h, n_buildings=5, n_trees=3, seed=0)
    g.mesh_to_phi(tris, objects, 2, out=torch.empty(g.shapes["phi"], dtype=g.torch_dtype, device="cuda"))


def use_transfers(g):
    fast = {n: torch.full(g.shapes[n], 50.0, dtype=g.torch_dtype).pin_memory() for n in ("u", "v", "w")}
    g.put_fields(fast)
    g.take_fields(fast)


def use_autotune(g):
    g.init_state()
    g.autotune(reps=1)
    g.set_tuning()


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("use", [use_mesh, use_transfers, use_autotune])
def test_initial_state_does_not_depend_on_earlier_calls(use, precision):
    sc = layouts.urban_block(40, 33, 12, h=2.0, n_boxes=3, n_trees=2, seed=6, footprint=(8.0, 14.0), height=(6.0, 14.0))
    out = []
    for before in (None, use):
        g = uf.Grid(sc.nx, sc.ny, sc.nz, precision=precision, **sc.params())
        if before:
            before(g)
        g.set_porosity(sc.phi.astype(g.np_dtype))
        g.init_state()
        dts = [g.step().dt for _ in range(2)]
        out.append((dts, g.state()))
    assert out[0][0] == out[1][0]
    for n in out[0][1]:
        np.testing.assert_array_equal(out[0][1][n], out[1][1][n], err_msg=n)
