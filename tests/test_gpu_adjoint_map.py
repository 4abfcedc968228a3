"""The adjoint's transpose map on bands whose nodes share sample cells by the hundred
(all samples drawn into few columns, so that a node's list of entries is long) and
on grids of a few chunks of the scan: the gradient against the transpose identity
<g, df> = <grad, dx> with the forward's own linearisation, by central differences
in FP64 (step 1e-6 of O(1) fields: truncation 1e-12, rounding 1e-10 of the sums,
so 1e-7 leaves a wide margin), and the same gradient from two handles bit for bit."""
import numpy as np
import pytest

from paper_2006_03343_gb300 import inputs

from parity_util import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def wm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_03343_gb300 import build, wmibm
    build.build()
    wmibm.load()
    return wmibm


def _funnel(shape):
    """A level set whose normals near the surface point towards one column: a steep
    cone, so that the sample points of many band nodes fall into a few cells."""
    nx, ny, nz = shape
    grid = (nx, ny, nz, 1.0, 1.0, 1.0)
    x = np.arange(nx) / nx - 0.5
    y = np.arange(ny) / ny - 0.5
    r = np.sqrt(x[None, :] ** 2 + y[:, None] ** 2)
    return grid, 0.75 - 0.6 * r


@pytest.mark.parametrize("shape", [(20, 18, 16), (40, 36, 24), (5, 7, 300), (130, 70, 9)])
@pytest.mark.parametrize("offset", [1.5, 6.0])
def test_gradient_by_central_differences(wm, shape, offset):
    grid, h2d = _funnel(shape)
    phi_uv, phi_w = inputs.heightfield_phi(grid, h2d)
    dz = 1.0 / (shape[2] - 1)
    rng = np.random.default_rng(3)
    make = lambda: wm.Handle(grid, phi_uv, phi_w, 1e-4, offset * dz, 0.5 * dz, dtype="f64")
    h = make()
    dims = (shape[2], shape[1], shape[0])
    vel = [rng.normal(1.0, 0.3, dims) for _ in range(3)]
    direction = [rng.normal(0.0, 1.0, dims) for _ in range(3)]
    tau = [to_dev(np.zeros(dims), "f64") for _ in range(6)]
    g = [to_dev(rng.normal(0.0, 1.0, dims), "f64") for _ in range(3)]

    def value(eps):
        f = [torch.zeros(dims, dtype=torch.float64, device="cuda") for _ in range(3)]
        h.wall_stress_force(*[to_dev(a + eps * d, "f64") for a, d in zip(vel, direction)], [t.clone() for t in tau], f)
        return sum(float((a * b).sum()) for a, b in zip(f, g))

    grads = []
    for handle in (h, make()):
        out = [torch.full(dims, float("nan"), dtype=torch.float64, device="cuda") for _ in range(4)]
        handle.backward(g, [to_dev(a, "f64") for a in vel], *out)
        grads.append(out)
    assert all(torch.equal(a, b) for a, b in zip(*grads))
    eps = 1e-6
    numeric = (value(eps) - value(-eps)) / (2 * eps)
    exact = sum(float((a * to_dev(d, "f64")).sum()) for a, d in zip(grads[0], direction))
    scale = sum(float((a * to_dev(d, "f64")).abs().sum()) for a, d in zip(grads[0], direction))
    assert abs(numeric - exact) <= 1e-7 * scale
