"""Step kernels whose threads march columns of several planes, at heights that
leave a remainder: an instance of a batch (always the full depth) equals the
same grid alone (a depth that fills the chip), bit for bit, and the step
equals its sub-steps run one by one."""
import numpy as np
import pytest

from paper_2204_01117_gb300 import layouts, uf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

# one plane, one more and one less than the depth, an odd height; ragged tiles; walls, inlets and outlets on every side
CASES = [((33, 9, 1), 30.0), ((32, 8, 7), 200.0), ((31, 17, 9), 135.0), ((65, 24, 18), 0.0)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uf.build()
    uf.load()


def scene(dims, deg):
    return layouts.urban_block(*dims, h=2.0, n_boxes=2, n_trees=2, seed=2, footprint=(4.0, 6.0), height=(2.0, 5.0),
                               wind_dir_deg=deg)


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_batch_equals_solo(precision):
    scenes = [scene(*c) for c in CASES]
    dims = lambda d: dict(zip(("nx", "ny", "nz"), d))
    b = uf.Batch([{**dims(d), **sc.params()} for (d, _), sc in zip(CASES, scenes)], precision=precision)
    for sc, g in zip(scenes, b.grids):
        g.set_porosity(sc.phi.astype(g.np_dtype))
        g.init_state()
    b.run(3)
    for (d, _), sc, gb in zip(CASES, scenes, b.grids):
        gs = uf.Grid(*d, precision=precision, **sc.params())
        gs.set_porosity(sc.phi.astype(gs.np_dtype))
        gs.init_state()
        gs.run(3)
        for f in ("u", "v", "w", "p", "k", "omega"):
            np.testing.assert_array_equal(gb.get_state(f), gs.get_state(f), err_msg=f"{d} {f}")


# 250 x 250 x 37: enough columns for the full depth in a grid alone
@pytest.mark.parametrize("dims, deg", CASES + [((250, 250, 37), 45.0)])
def test_step_equals_sub_steps(dims, deg):
    sc = scene(dims, deg)
    params = {**sc.params(), "fixed_dt": 0.2}
    g = uf.Grid(*dims, precision="f64", **params)
    g.set_porosity(sc.phi)
    g.init_state()
    g.run(2)
    s = g.state()
    nut, = g.substep("eddy", [s[n] for n in ("u", "v", "w", "k", "omega")])
    u2 = g.substep("diffuse", g.substep("advect", [s[n] for n in "uvw"]) + [nut])
    u1 = g.substep("project", g.substep("drag_bc", u2 + [sc.phi]))
    k1, o1 = g.substep("turb", u1 + [s["k"], s["omega"]])
    ref = uf.Grid(*dims, precision="f64", **params)
    ref.set_porosity(sc.phi)
    ref.set_fields({n: s[n] for n in ("u", "v", "w", "k", "omega")})
    ref.step()
    # two solves to the default tolerance
    for name, got in zip(("u", "v", "w", "k", "omega"), u1 + [k1, o1]):
        r = ref.get_state(name)
        assert np.linalg.norm(got - r) <= 1e-9 * np.linalg.norm(r), name
