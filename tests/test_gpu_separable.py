"""The separable inverse that grids use as their default preconditioner
(csrc/sep_solve.cuh): the pressure solve against a direct FP64 solve (numpy
eigenvectors of the three axis matrices) at the edges of its panels and
lines, and whole steps against the V-cycle (coarse_start = -1) it replaces.

Tolerance of the solve: 5e-5, the bound of the other FP32 pressure solves
(||r|| <= 1e-7 ||b|| and a random right-hand side of N cells leave at most
1e-7 sqrt(N), 5e-5 at N = 250 000); FP64 likewise 1e-9, ||r|| <= 1e-12 ||b||."""
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


def direct_solve(b, deg):
    c, s = np.cos(np.radians(deg)), np.sin(np.radians(deg))
    out = [(c < -1e-9, c > 1e-9), (s < -1e-9, s > 1e-9), (False, False)]   # outlet at the low / high end of x, y, z
    lam, vec = [], []
    for n, (lo, hi) in zip(b.shape[::-1], out):
        T = 2.0 * np.eye(n) - np.eye(n, k=1) - np.eye(n, k=-1)
        T[0, 0] -= not lo
        T[-1, -1] -= not hi
        w, q = np.linalg.eigh(T)
        lam.append(w)
        vec.append(q)
    t = np.einsum("kji,kc,jb,ia->cba", b, vec[2], vec[1], vec[0], optimize=True)
    t /= lam[2][:, None, None] + lam[1][None, :, None] + lam[0][None, None, :]
    return np.einsum("cba,kc,jb,ia->kji", t, vec[2], vec[1], vec[0], optimize=True)


# one value per lane to 32, odd panels of x, ny past one shared-memory panel (768), nz = 1, 2 and past a 64-row round
@pytest.mark.parametrize("dims, deg", [((2, 2, 1), 0.0), ((5, 3, 2), 200.0), ((33, 45, 9), 300.0), ((64, 70, 1), 180.0),
                                       ((97, 16, 17), 90.0), ((130, 65, 70), 45.0), ((260, 9, 5), 270.0), ((513, 12, 3), 0.0),
                                       ((1024, 4, 2), 135.0), ((6, 769, 2), 30.0), ((40, 768, 1), 90.0), ((7, 1392, 1), 10.0),
                                       ((9, 8, 400), 60.0),
                                       # folded in y too: odd halves, one cell past a 16-row tile, the widest panel
                                       ((40, 37, 21), 0.0), ((12, 33, 34), 180.0), ((32, 761, 3), 0.0), ((8, 1391, 1), 180.0)])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_solve_matches_direct(dims, deg, precision):
    nx, ny, nz = dims
    b = np.random.default_rng(nx + ny).standard_normal((nz, ny, nx))
    g = uf.Grid(nx, ny, nz, precision=precision, wind_dir_deg=deg)
    assert g.get_tuning()[0]["coarse_start"] == (0 if precision == "f32" or ny + nz <= 480 else -1)
    g.set_state("p", 0.0)
    b = b.astype(g.np_dtype)
    it, r = g.poisson_solve(b)
    ref = direct_solve(b.astype(np.float64), deg)
    assert r <= (1e-7 if precision == "f32" else 1e-12)
    assert it <= 5 or g.get_tuning()[0]["coarse_start"] == -1, it
    assert np.linalg.norm(g.get_state("p") - ref) <= (5e-5 if precision == "f32" else 1e-9) * np.linalg.norm(ref)


def test_other_requests_keep_the_v_cycle():
    for precision in ("f32", "f64"):
        for kw in (dict(mg_smoother="rbgs"), dict(mg_transfer="constant")):
            g = uf.Grid(32, 24, 12, precision=precision, **kw)
            assert g.get_tuning()[0]["coarse_start"] == -1
        assert uf.Grid(32, 24, 12, precision=precision).get_tuning()[0]["coarse_start"] == 0
    assert uf.Grid(4, 440, 40, precision="f64").get_tuning()[0]["coarse_start"] == 0
    assert uf.Grid(4, 440, 41, precision="f64").get_tuning()[0]["coarse_start"] == -1
    g = uf.Grid(32, 24, 12)
    g.set_tuning(coarse_start=-1)
    assert g.get_tuning()[0]["coarse_start"] == -1
    for dims in ((1025, 4, 2), (4, 1393, 2), (4, 4, 401)):
        assert uf.Grid(*dims).get_tuning()[0]["coarse_start"] == -1


def test_switching_there_and_back():
    """The V-cycle overwrites the pivots' memory; a grid that returns to the separable inverse steps as one that never left."""
    sc = layouts.urban_block(40, 33, 12, h=2.0, n_boxes=3, n_trees=2, seed=6, footprint=(8.0, 14.0), height=(6.0, 14.0))
    out = []
    for detour in (False, True):
        g = uf.Grid(sc.nx, sc.ny, sc.nz, **sc.params())
        g.set_porosity(sc.phi.astype(np.float32))
        g.init_state()
        if detour:
            keep = g.save_checkpoint()
            g.set_tuning(coarse_start=-1)
            g.run(2)
            g.set_tuning()
            g.load_checkpoint(keep)
        g.run(2)
        out.append(g.state())
    for n in out[0]:
        np.testing.assert_array_equal(out[0][n], out[1][n], err_msg=n)


@pytest.mark.parametrize("precision", ["f32", "f64"])
@pytest.mark.parametrize("deg", [0.0, 120.0, 270.0])
def test_steps_match_the_v_cycle(deg, precision):
    sc = layouts.urban_block(61, 47, 19, h=2.0, n_boxes=4, n_trees=4, seed=3, footprint=(8.0, 20.0), height=(6.0, 24.0),
                             wind_dir_deg=deg)
    out = []
    for cs in (0, -1):
        g = uf.Grid(sc.nx, sc.ny, sc.nz, precision=precision, **sc.params())
        g.set_tuning(coarse_start=cs)
        g.set_porosity(sc.phi.astype(g.np_dtype))
        g.init_state()
        assert g.run(3).status == 0
        out.append(g.state())
    for n in out[0]:
        assert np.linalg.norm(out[0][n] - out[1][n]) <= (1e-5 if precision == "f32" else 1e-10) * np.linalg.norm(out[1][n]), n


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_batch_mixes_both(precision):
    """An instance with the V-cycle asked for beside two that use the separable inverse: each as it computes alone."""
    insts = [dict(nx=48, ny=40, nz=12, u_ref=3.0), dict(nx=64, ny=33, nz=9, u_ref=4.0, wind_dir_deg=70.0), dict(nx=40, ny=24, nz=16, u_ref=2.0)]
    phi = [np.random.default_rng(q).random((p["nz"], p["ny"], p["nx"])).astype(np.float32) * 0.5 + 0.5 for q, p in enumerate(insts)]
    b = uf.Batch(insts, precision=precision)
    solos = [uf.Grid(precision=precision, **p) for p in insts]
    for q in range(3):
        for g in (b.grids[q], solos[q]):
            if q == 1:
                g.set_tuning(coarse_start=-1)
            g.set_porosity(phi[q].astype(g.np_dtype))
            g.init_state()
    b.run(3)
    for q, g in enumerate(solos):
        g.run(3)
        for f in ("u", "v", "w", "p", "k", "omega"):
            np.testing.assert_array_equal(b.grids[q].get_state(f), g.get_state(f), err_msg=f"{q} {f}")
