"""The eddy factor -2 sqrt(q) / L of the FP32 tile march, element by element against 64
bits, over the window that its Newton step takes, the window's edges and beyond, where
the plain operations take over: zero, tiny, huge, infinite and NaN strains.

The velocity depends on z alone and dx = dy = dz = 1/8, so that a w-node's only strain is
S13 and q = (2 S13)^2; L = lam + wall term with wall terms drawn over the exponents, and
lam = 64 / cs^2 small.  tau_xz = factor * S13.

Tolerances, in units u = 2^-24 of the exact value.  In the window the factor is off by
(1 + 2^-17) u (half an ulp and what the Newton step leaves) and the product adds u:
2.001 u.  The plain operations round three times with the product, and so do four x-neighbours
of which one is off the window: 4.001 u (a root, a quotient and a product: 3 u, and
second-order terms).  Where the plain operations leave the normal range the result is that of
the same operations in FP32 on the host (NaN, infinities) or off by two of the smallest numbers."""
import numpy as np
import pytest

from paper_2006_03343_gb300 import inputs

from parity_util import to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPE = (32, 16, 9)                 # nx, ny, nz
U = 2.0 ** -24
CS = 2.0 ** 23                      # 1 / lambda_0^2 = (8 / CS)^2 = 2^-40


@pytest.fixture(scope="module")
def setup():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_03343_gb300 import build, wmibm
    build.build()
    wmibm.load()
    nx, ny, nz = SHAPE
    case = inputs.flat(SHAPE, wall_height=-1.0, lengths=(nx / 8, ny / 8, 1.0))
    return wmibm.Handle.from_case(case, dtype="f32")


def _stress(h, levels, wt, cs=CS):
    """tau_xz for u(k) = levels[k] and wall terms wt, both FP32."""
    shape = h.shape
    u = torch.from_numpy(np.ascontiguousarray(np.broadcast_to(levels[:, None, None], shape))).cuda()
    zero = torch.zeros_like(u)
    w = torch.from_numpy(wt).cuda()
    tau = [torch.zeros_like(u) for _ in range(6)]
    h.sgs_stress(u, zero, zero, (w, w), tau, cs=cs)
    return tau[4].cpu().numpy()


def _factors(levels, wt):
    """S13, q and L at the inner w-levels as the kernel rounds them."""
    s13 = (levels[1:-1] - levels[:-2]) * np.float32(4.0)            # 1 / (2 dz)
    d = np.float32(2.0) * s13
    return s13[:, None, None], (d * d)[:, None, None], np.float32(2.0 ** -40) + wt[1:-1]


def _in_window(q, L):
    inside = (q >= 2.0 ** -60) & (q < 2.0 ** 40) & (L >= 2.0 ** -30) & (L < 2.0 ** 43)
    return np.repeat(inside.reshape(*L.shape[:2], -1, 4).all(axis=-1), 4, axis=-1)


@pytest.mark.parametrize("seed", range(4))
def test_factor_over_the_exponents(setup, seed):
    h = setup
    rng = np.random.default_rng(seed)
    worst, checked = [0.0, 0.0], 0
    with np.errstate(all="ignore"):
        for e in range(-75, 64):
            levels = (rng.uniform(-1.0, 1.0, h.shape[0]) * 2.0 ** e).astype(np.float32)
            # half the nodes within the window of L, half of them at its edges and beyond
            exps = rng.uniform(-30.0, 43.0, h.shape) if rng.random() < 0.5 else rng.uniform(-36.0, 60.0, h.shape)
            wt = (2.0 ** exps).astype(np.float32)
            s13, q, L = _factors(levels, wt)
            got = _stress(h, levels, wt)[1:-1].astype(np.float64)
            plain = (np.float32(-2.0) * np.sqrt(q)) / L
            f32 = plain * s13
            exact = -2.0 * np.sqrt(q.astype(np.float64)) / L.astype(np.float64) * s13.astype(np.float64)
            inside = _in_window(q, L)
            tiny = np.finfo(np.float32).tiny
            normal = np.isfinite(f32) & (np.abs(plain) >= tiny) & (np.abs(exact) >= 2 * tiny) & (q >= tiny)
            err = np.abs(got - exact) / np.where(exact == 0.0, 1.0, np.abs(exact)) / U
            assert np.all(normal[inside])
            for n, (mask, tol) in enumerate(((inside, 2.001), (~inside & normal, 4.001))):
                if mask.any():
                    worst[n] = max(worst[n], float(err[mask].max()))
                    assert err[mask].max() <= tol, (e, n, worst)
            rest = ~inside & ~normal
            assert np.all(np.abs(got - f32.astype(np.float64))[rest & np.isfinite(f32)] <= 2 * 2.0 ** -149 + 4 * U * tiny)
            assert np.array_equal(got[~np.isfinite(f32)], f32[~np.isfinite(f32)].astype(np.float64), equal_nan=True)
            checked += int(inside.sum())
    assert checked > 50000
    print(worst)


@pytest.mark.parametrize("step", [0.0, -0.0, 2.0 ** -149, 2.0 ** 64, 3e38, np.inf, -np.inf, np.nan])
def test_special_strains(setup, step):
    h = setup
    rng = np.random.default_rng(9)
    levels = np.zeros(h.shape[0], np.float32)
    levels[5:] = np.float32(step)           # between levels 4 and 5 alone
    wt = (2.0 ** rng.uniform(-20.0, 20.0, h.shape)).astype(np.float32)
    with np.errstate(all="ignore"):
        s13, q, L = _factors(levels, wt)
        f32 = (np.float32(-2.0) * np.sqrt(q)) / L * s13
    if not np.isfinite(step):
        f32[4:] = np.nan                    # the x differences of infinities are NaN, and q with them
    got = _stress(h, levels, wt)[1:-1]
    assert np.array_equal(np.isnan(got), np.isnan(f32))
    both = ~np.isnan(f32)
    assert np.array_equal(np.isinf(got[both]), np.isinf(f32[both]))
    finite = np.isfinite(f32)
    err = np.abs(got[finite].astype(np.float64) - f32[finite].astype(np.float64))
    assert np.all(err <= 8 * U * np.abs(f32[finite]) + 4 * 2.0 ** -149)


def test_quotient_beyond_the_range(setup):
    """sqrt(q) / L overflows although q and L are ordinary: -inf, as by the plain operations."""
    h = setup
    levels = np.zeros(h.shape[0], np.float32)
    levels[5:] = np.float32(2.0 ** 46)      # q = 2^98 at one w-level
    wt = np.full(h.shape, 2.0 ** -90, np.float32)
    got = _stress(h, levels, wt, cs=2.0 ** 50)
    assert np.all(got[5] == -np.inf)
    assert np.all(got[1:5] == 0.0) and np.all(got[6:-1] == 0.0)
