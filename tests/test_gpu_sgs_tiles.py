"""The SGS tile march (k_sgs_tile) at the edges of its tiles, against the FP64
oracle: rows that fit a warp whole (nx <= 128, one to 32 lanes), rows cut into
tiles with halo lanes, rows that no vector divides, tiles of fewer rows than a
block holds, chunks of levels down to the minimal grid, and zero velocity (the
plain square root).  The tolerance is the one of every FP32 / FP64 comparison
with the oracle: 1e-5 and 1e-12 of the array's largest value."""
import numpy as np
import pytest

from paper_2006_03343_gb300 import inputs

from parity_util import TOL, normwise, to_dev, to_host

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CS = 0.16
SHAPES = [(4, 3, 3), (8, 33, 5), (20, 14, 9), (64, 15, 17), (124, 7, 12), (128, 13, 20), (132, 29, 11), (260, 31, 18),
          (5, 16, 4), (57, 28, 9), (113, 6, 13), (130, 17, 40)]


@pytest.fixture(scope="module")
def wm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_03343_gb300 import build, wmibm
    build.build()
    wmibm.load()
    return wmibm


def _compare(wm, oracle_mod, case, dtype, vel):
    h = wm.Handle.from_case(case, dtype=dtype, vel_dtype=vel)
    wt = h.sgs_wall_terms(case.phi_uv, case.phi_w, case.z0)
    vd = vel or dtype
    u, v, w = (to_dev(x, vd) for x in (case.u, case.v, case.w))
    ref = {k: to_host(to_dev(case.tau[k], dtype)) for k in inputs.TAU_NAMES}
    tau = [to_dev(case.tau[k], dtype) for k in inputs.TAU_NAMES]
    h.sgs_stress(u, v, w, wt, tau, cs=CS)
    rv = lambda a: to_host(to_dev(a, vd))
    oracle_mod.sgs_stress(case.grid, case.phi_uv, case.phi_w, case.z0, case.phi_b, rv(case.u), rv(case.v), rv(case.w),
                          ref, cs=CS, kappa=inputs.KAPPA)
    for k, t in zip(inputs.TAU_NAMES, tau):
        assert normwise(to_host(t), ref[k])[0] <= TOL[dtype], k
    tau = [to_dev(case.tau[k], dtype) for k in inputs.TAU_NAMES]
    f = [torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda") for _ in range(3)]
    h.wall_stress(u, v, w, tau)
    h.sgs_force(u, v, w, wt, tau, f, cs=CS)
    oracle_mod.wall_stress(case.grid, case.phi_uv, case.phi_w, case.z0, case.phi_c, case.phi_b, rv(case.u), rv(case.v),
                           rv(case.w), ref)
    for got, want in zip(f, oracle_mod.force(case.grid, ref)):
        got = to_host(got)
        assert np.all(np.isfinite(got))
        assert normwise(got, want)[0] <= TOL[dtype]


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("dtype,vel", [("f32", None), ("f32", "bf16"), ("f64", None)])
def test_tile_edges_match_the_oracle(wm, oracle_mod, shape, dtype, vel):
    case = inputs.flat(shape, wall_height=0.21, lengths=(2.0, 1.5, 1.0), sigma=0.1, seed=7)
    _compare(wm, oracle_mod, case, dtype, vel)


def test_zero_velocity_gives_zero_stress(wm):
    case = inputs.flat((64, 20, 12), wall_height=0.21, sigma=0.1, seed=3)
    h = wm.Handle.from_case(case, dtype="f32")
    wt = h.sgs_wall_terms(case.phi_uv, case.phi_w, case.z0)
    u = [torch.zeros(h.shape, device="cuda") for _ in range(3)]
    tau = [torch.zeros(h.shape, device="cuda") for _ in range(6)]
    f = [torch.full(h.shape, float("nan"), device="cuda") for _ in range(3)]
    h.sgs_stress(*u, wt, tau, cs=CS)
    h.sgs_force(*u, wt, tau, f, cs=CS)
    assert all(float(t.abs().max()) == 0.0 for t in tau + f)
