"""The sigmoid design map and its transpose at the edges of their tiles (32 x
8 columns, 8 planes) and at both ends of the number of boxes, with boxes that
reach no cell, one tile, and all of them."""
import numpy as np
import pytest

import oracle
from paper_2204_01117_gb300 import uf

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
H = 2.0


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    uf.build()
    uf.load()
    oracle.build()


def setup(dims, nbox, seed):
    """Boxes over the whole domain and past its ends (every fourth one far
    outside, so that it reaches no cell)."""
    rng = np.random.default_rng(seed)
    nx, ny, _ = dims
    boxes, theta = [], []
    for b in range(nbox):
        x, y = rng.uniform(-4, nx * H), rng.uniform(-4, ny * H)
        if b % 4 == 3:
            x += 1e4
        boxes.append((x, x + rng.uniform(1, 30), y, y + rng.uniform(1, 30)))
        theta += [rng.uniform(0.0, 2 * dims[2]), rng.uniform(-3, 3), rng.uniform(-3, 3)]
    return boxes, np.array(theta)


def reference_vjp(dims, boxes, theta, width, lam):
    """Gradient of sum(lam * phi) by automatic differentiation in FP64."""
    nx, ny, nz = dims
    t = torch.tensor(theta, dtype=torch.float64, requires_grad=True)
    x, y, z = ((torch.arange(n, dtype=torch.float64) + 0.5) * H for n in (nx, ny, nz))
    s = lambda a: torch.sigmoid(a / width)
    phi = torch.ones(nz, ny, nx, dtype=torch.float64)
    for b, (xa, xb, ya, yb) in enumerate(boxes):
        hh, dx, dy = t[3 * b], t[3 * b + 1], t[3 * b + 2]
        cx, cy, cz = s(x - (xa + dx)) * s((xb + dx) - x), s(y - (ya + dy)) * s((yb + dy) - y), s(hh - z)
        phi = phi * (1 - cz[:, None, None] * cy[None, :, None] * cx[None, None, :])
    (phi * torch.tensor(lam)).sum().backward()
    return t.grad.numpy()


# widths: sharp ramps (a box leaves most tiles at exactly 1) and one wider than the domain
@pytest.mark.parametrize("dims, nbox, width", [((33, 9, 9), 5, 0.05), ((32, 8, 8), 1, 1.0), ((31, 7, 1), 2, 2.0),
                                               ((70, 25, 17), 64, 0.5), ((40, 16, 7), 64, 200.0)])
@pytest.mark.parametrize("precision", ["f32", "f64"])
def test_map_and_transpose(dims, nbox, width, precision):
    boxes, theta = setup(dims, nbox, nbox)
    g = uf.Grid(*dims, h=H, precision=precision)
    ref = oracle.design_to_phi(*dims, H, boxes, theta, width)
    # ramps of a coordinate of up to 140 m, rounded to 2e-14 m: 1e-13 of a ramp of width 0.05 m, a few ramps
    # near their edge at a cell; FP32: one rounding of the FP64 value
    np.testing.assert_allclose(g.design_to_phi(boxes, theta, width, set_porosity=False), ref, rtol=0,
                               atol=1e-12 if precision == "f64" else 1e-7)
    lam = np.random.default_rng(1).standard_normal(g.shapes["phi"]).astype(g.np_dtype)
    want = reference_vjp(dims, boxes, theta, width, lam.astype(np.float64))
    got = g.design_vjp(boxes, theta, width, lam)
    # sums of up to 30000 terms of at most 1 / width, 1e-15 each: 1e-12 of the sum of their magnitudes
    np.testing.assert_allclose(got, want, rtol=1e-12, atol=1e-12 * lam.size / width)
