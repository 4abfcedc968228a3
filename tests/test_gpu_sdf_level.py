"""wmibm_heightfield_sdf where many triangles tie: nearly level ground (slopes from
1e-2 down to below the ulp of a distance), gentle planes in every direction,
valleys, ridges, peaks and pits at a vertex, and cells of unequal sides, against
the oracle's brute force.  The tolerance is that of the other distance tests:
1e-12, some hundred ulps of the lengths involved."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

TOL = 1e-12
EDGE = 1e-9


@pytest.fixture(scope="module")
def wm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_03343_gb300 import build, wmibm
    build.build()
    wmibm.load()
    return wmibm


def _terrain(kind, nx, ny, lx, ly, size):
    x = np.arange(nx) * (2 * np.pi / nx)
    y = np.arange(ny) * (2 * np.pi / ny)
    i, j = np.meshgrid(np.arange(nx), np.arange(ny))
    wave = np.sin(x)[None, :] * 0.7 + np.cos(y)[:, None] * 0.4
    if kind == "waves":
        return 0.3 + size * wave
    if kind == "creases":       # valleys and ridges along x, y and the diagonal
        return 0.3 + size * (np.abs((i % 6) - 3) + np.abs((j % 4) - 2) - np.abs(((i - j) % 8) - 4))
    h = np.full((ny, nx), 0.3)  # peaks and pits
    h[::4, ::3] += size
    h[2::4, 1::3] -= 0.5 * size
    return h


@pytest.mark.parametrize("kind", ["waves", "creases", "points"])
@pytest.mark.parametrize("size", [3e-2, 1e-4, 1e-7, 1e-11, 1e-16])
@pytest.mark.parametrize("lengths", [(1.0, 1.0), (1.7, 0.6)])
def test_nearly_level_ground_matches_the_oracle(wm, oracle_mod, kind, size, lengths):
    nx, ny, nz = 36, 24, 22
    grid = (nx, ny, nz) + lengths + (1.0,)
    h = _terrain(kind, nx, ny, *lengths, size)
    reach = 2.6 / (nz - 1)
    pu, pw = wm.heightfield_sdf(grid, torch.from_numpy(h).cuda(), reach)
    torch.cuda.synchronize()
    dz = 1.0 / (nz - 1)
    for is_w, got in ((False, pu), (True, pw)):
        d = oracle_mod.heightfield_distance(grid, h, is_w, None)
        z = (np.arange(nz) + (0.0 if is_w else 0.5)) * dz
        vert = z[:, None, None] - h[None]
        ref = np.where(d <= reach, np.copysign(d, vert), vert)
        away = np.abs(d - reach) > EDGE
        assert np.max(np.abs(got.cpu().numpy() - ref)[away]) <= TOL
