"""The transpose of the design map for boxes far from every sensitivity: their
gradients are tiny, not zero, and a sensitivity that is not a number reaches
every box."""
import numpy as np
import pytest

from paper_2204_01117_gb300 import uf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
H, WIDTH, DIMS = 2.0, 1.0, (64, 48, 24)
# 90 ramp widths west of the sensitivities below, 10 km away (chi = 0), among them
BOXES = [(10.0, 30.0, 13.0, 37.0), (1e4, 1e4 + 20.0, 20.0, 40.0), (112.0, 124.0, 70.0, 84.0)]
THETA = np.array([20.0, 0.3, -0.2, 30.0, 0.0, 0.0, 25.0, -0.4, 0.5])


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uf.build()
    uf.load()


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_gradient_of_a_distant_box(precision):
    g = uf.Grid(*DIMS, h=H, precision=precision)
    lam = np.zeros(g.shapes["phi"], dtype=g.np_dtype)
    lam[:, 30:, 60:] = np.random.default_rng(0).uniform(0.5, 1.5, (24, 18, 4))   # east and north of the first box
    t = torch.tensor(THETA, dtype=torch.float64, requires_grad=True)
    x, y, z = ((torch.arange(n, dtype=torch.float64) + 0.5) * H for n in DIMS)
    s = lambda a: torch.sigmoid(a / WIDTH)
    phi = torch.ones(lam.shape, dtype=torch.float64)
    for b, (xa, xb, ya, yb) in enumerate(BOXES):
        hh, dx, dy = t[3 * b], t[3 * b + 1], t[3 * b + 2]
        cx, cy = s(x - (xa + dx)) * s((xb + dx) - x), s(y - (ya + dy)) * s((yb + dy) - y)
        phi = phi * (1 - s(hh - z)[:, None, None] * cy[None, :, None] * cx[None, None, :])
    (phi * torch.tensor(lam.astype(np.float64))).sum().backward()
    want = t.grad.numpy()
    got = g.design_vjp(BOXES, THETA, WIDTH, lam)
    assert 0 < abs(want[0]) < 1e-40 and 0 < abs(want[1]) < 1e-40 and 0 < abs(want[2]) < 1e-40, want[:3]
    # terms of one sign; ramp arguments of up to 130 widths, rounded to 3e-14
    np.testing.assert_allclose(got[:3], want[:3], rtol=1e-12, atol=0)
    np.testing.assert_array_equal(got[3:6], 0.0)
    np.testing.assert_allclose(got[6:], want[6:], rtol=1e-10, atol=1e-12 * lam.size)


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_a_nan_reaches_every_box(precision):
    g = uf.Grid(*DIMS, h=H, precision=precision)
    lam = np.zeros(g.shapes["phi"], dtype=g.np_dtype)
    lam[3, 40, 63] = np.nan
    assert np.isnan(g.design_vjp(BOXES, THETA, WIDTH, lam)).all()


@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_a_nan_parameter_stays_with_the_sensitivities(precision):
    """A box whose height is not a number: every gradient is, where there are sensitivities, and 0 where there are none."""
    g = uf.Grid(*DIMS, h=H, precision=precision)
    theta = THETA.copy()
    theta[6] = np.nan
    lam = np.zeros(g.shapes["phi"], dtype=g.np_dtype)
    np.testing.assert_array_equal(g.design_vjp(BOXES, theta, WIDTH, lam), 0.0)
    lam[3, 40, 60] = 1.0
    assert np.isnan(g.design_vjp(BOXES, theta, WIDTH, lam)).all()
