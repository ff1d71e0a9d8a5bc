"""Tuning a grid or a batch leaves its automatic choices in force."""
import pytest

from paper_2204_01117_gb300 import uf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uf.build()
    uf.load()


def advect_us(x, label):
    """Least time of the advection in a few eagerly launched steps."""
    def once():
        r = x.profile_step()
        return (r[1] if isinstance(r, tuple) else r)[label]["total_ms"] * 1e3
    return min(once() for _ in range(8))


# A grid of 48 x 40 x 16 advects with one plane per block in 12 us and with 16 in 44 us: a factor of two tells them apart.

def round_trip(g):
    g.set_tuning(**g.get_tuning()[0])


@pytest.mark.parametrize("tune", [lambda g: g.autotune(reps=1), round_trip], ids=["autotune", "round trip"])
def test_a_tuned_grid_keeps_the_automatic_advection_depth(tune):
    g = uf.Grid(48, 40, 16)
    g.init_state()
    before = advect_us(g, "advect_fused")
    tune(g)
    assert g.get_tuning()[0]["advect_zc"] == 16
    assert advect_us(g, "advect_fused") < 2 * before


def test_a_tuned_batch_keeps_the_automatic_advection_depth():
    b = uf.Batch([dict(nx=48, ny=40, nz=16), dict(nx=40, ny=32, nz=20)])
    for g in b.grids:
        g.init_state()
    before = advect_us(b, "b_advect_fused")
    b.autotune(reps=1)
    assert advect_us(b, "b_advect_fused") < 2 * before


def test_an_explicit_advection_depth_stays():
    g = uf.Grid(48, 40, 16)
    g.init_state()
    before = advect_us(g, "advect_fused")
    for depth in (15, 17):
        g.set_tuning(advect_zc=depth)
        g.autotune(reps=1)
        assert g.get_tuning()[0]["advect_zc"] == depth
        assert advect_us(g, "advect_fused") > 2 * before


@pytest.mark.parametrize("order", [0, 1])
def test_a_batch_does_not_share_a_tuning_across_solvers(order):
    """Grids of one size, of which only the second can use the separable inverse: each is tuned for its own solver.
    (On 40 x 32 x 16 the inverse wins the tuning by a factor of three.)"""
    size = dict(nx=40, ny=32, nz=16)
    insts = [dict(size, mg_transfer="constant"), size]
    b = uf.Batch(insts[::-1] if order else insts)
    assert b.autotune(reps=1) == 2
    plain, capable = b.grids[::-1] if order else b.grids
    assert plain.get_tuning()[0]["coarse_start"] != 0
    assert capable.get_tuning()[0]["coarse_start"] == 0
    for g in b.grids:
        g.init_state()
    b.run(2)


# both sides of the rule that uf.h states for coarse_start = 0 (the edges of single axes: test_gpu_separable.py)
@pytest.mark.parametrize("dims, precision, inverse", [((1024, 256, 4), "f64", True), ((1024, 257, 4), "f64", False),
                                                      ((993, 257, 4), "f64", False), ((992, 264, 4), "f64", True),
                                                      ((1024, 257, 1), "f64", True), ((1024, 991, 2), "f32", True)])
def test_the_stated_size_rule(dims, precision, inverse):
    assert uf.Grid(*dims, precision=precision).get_tuning()[0]["coarse_start"] == (0 if inverse else -1)
