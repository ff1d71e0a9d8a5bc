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
