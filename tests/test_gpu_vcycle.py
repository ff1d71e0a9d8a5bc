"""The V-cycle with the default smoother and transfers, which grids past the
sizes of the separable inverse run: asked for here (coarse_start = -1) at sizes
where the inverse would otherwise take its place."""
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest

from paper_2204_01117_gb300 import layouts, uf
from test_gpu_separable import direct_solve

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
FIELDS = ("u", "v", "w", "p", "k", "omega")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uf.build()
    uf.load()


def vcycle(nx, ny, nz, tuning=None, **kw):
    g = uf.Grid(nx, ny, nz, **kw)
    g.set_tuning(**dict(dict(coarse_start=-1), **(tuning or {})))
    assert g.get_tuning()[0]["coarse_start"] != 0
    return g


# as the other FP32 and FP64 pressure solves: ||r|| <= 1e-7 (1e-12) ||b|| of a random right-hand side
@pytest.mark.parametrize("dims, deg", [((48, 40, 16), 0.0), ((57, 43, 21), 30.0), ((130, 65, 33), 225.0), ((64, 70, 1), 90.0)])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_solve_matches_direct(dims, deg, precision):
    nx, ny, nz = dims
    g = vcycle(nx, ny, nz, precision=precision, wind_dir_deg=deg)
    b = np.random.default_rng(nx).standard_normal((nz, ny, nx)).astype(g.np_dtype)
    g.set_state("p", 0.0)
    it, r = g.poisson_solve(b)
    ref = direct_solve(b.astype(np.float64), deg)
    assert 5 < it <= 60 and r <= (1e-7 if precision == "f32" else 1e-12), (it, r)   # (the inverse takes at most 5)
    assert np.linalg.norm(g.get_state("p") - ref) <= (5e-5 if precision == "f32" else 1e-9) * np.linalg.norm(ref)


def scene(seed=0):
    return layouts.urban_block(64, 56, 24, h=2.0, n_boxes=4, n_trees=4, seed=seed, footprint=(8.0, 20.0), height=(6.0, 24.0))


def started(sc, tuning=None):
    g = vcycle(sc.nx, sc.ny, sc.nz, tuning=tuning, **sc.params())
    g.set_porosity(sc.phi.astype(np.float32))
    g.init_state()
    return g


def test_tail_and_tile_depth_give_the_same_step():
    sc = scene()
    g = started(sc)
    g.run(2)
    before = g.state()
    levels = g.get_tuning()[1]
    for tuning in (dict(tail_level=levels - 1, march_zc=[2] * 16), dict(march_zc=[8] * 16), dict(coarse_start=1)):
        h = vcycle(sc.nx, sc.ny, sc.nz, tuning=tuning, **sc.params())
        h.set_porosity(sc.phi.astype(np.float32))
        h.set_fields(before)
        g.set_fields(before)
        g.run(1)
        h.run(1)
        for f in FIELDS:   # the same up to the order of FP64 sums
            a, r = h.get_state(f).astype(np.float64), g.get_state(f).astype(np.float64)
            assert np.linalg.norm(a - r) <= 1e-5 * max(np.linalg.norm(r), 1e-30), (tuning, f)


def test_grids_with_different_tails_coexist():
    """The tail kernel's shared-memory limit is per kernel: a grid with a smaller tail that comes later must not break the
    graphs of one with a larger."""
    big, small = vcycle(48, 40, 12), vcycle(24, 20, 8)
    for g in (big, small):
        g.init_state()
    for g in (big, small, big):
        g.run(2)


def test_a_batch_equals_its_grids_alone():
    scs = [scene(1), layouts.urban_block(48, 40, 16, h=2.0, seed=2)]
    b = uf.Batch([dict(nx=s.nx, ny=s.ny, nz=s.nz, **s.params()) for s in scs])
    for s, g in zip(scs, b.grids):
        g.set_tuning(coarse_start=-1)
        g.set_porosity(s.phi.astype(np.float32))
        g.init_state()
    b.run(3)
    for s, gb in zip(scs, b.grids):
        g = started(s)
        g.run(3)
        for f in FIELDS:
            np.testing.assert_array_equal(gb.get_state(f), g.get_state(f), err_msg=f)


CHILD = textwrap.dedent("""
    import os, sys
    import numpy as np
    sys.path.insert(0, os.environ["UF_ROOT"])
    from paper_2204_01117_gb300 import layouts, uf
    assert uf.load().uf_bounds_checked() == 1
    sc = layouts.urban_block(70, 54, 19, h=2.0, seed=2, wind_dir_deg=200.0)
    for precision in ("f32", "f64"):
        g = uf.Grid(sc.nx, sc.ny, sc.nz, precision=precision, **sc.params())
        g.set_tuning(coarse_start=-1)
        g.set_porosity(sc.phi.astype(g.np_dtype))
        g.init_state()
        g.run(3)
        g.close()
    insts = [layouts.urban_block(n, m, k, h=2.0, seed=s) for (n, m, k, s) in ((48, 40, 16, 1), (36, 30, 12, 2), (41, 33, 9, 3))]
    bt = uf.Batch([dict(nx=x.nx, ny=x.ny, nz=x.nz, **x.params()) for x in insts], precision="f32")
    for x, gi, cs in zip(insts, bt.grids, (-1, 0, -1)):   # both solvers in one batch
        gi.set_tuning(coarse_start=cs)
        gi.set_porosity(x.phi.astype(np.float32))
        gi.init_state()
    bt.run(3)
    bt.close()
    print("clean")
""")


def test_bounds_checked_build_runs_it_clean():
    env = dict(os.environ, UF_LIBRARY=uf.build(checked=True), UF_ROOT=ROOT)
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, capture_output=True, text=True, timeout=1500)
    assert r.returncode == 0 and "clean" in r.stdout, r.stdout[-3000:] + r.stderr[-3000:]
