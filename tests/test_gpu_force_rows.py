"""The direct-load forcing at the row lengths and alignments between which it
chooses its vectors (two values where rows and buffers are 8-byte aligned, one
otherwise), and the wall kernel's launch for bands from none to many per SM,
against the FP64 oracle: 1e-5 of each array's largest value in FP32, 1e-12 in FP64."""
import numpy as np
import pytest

from paper_2006_03343_gb300 import inputs

from parity_util import TOL, normwise, to_dev, to_host

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


def _shifted(t, shift):
    buf = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)
    return buf[shift:].view(t.shape).copy_(t)


@pytest.mark.parametrize("nx", [1, 2, 6, 62, 65, 66, 130])
@pytest.mark.parametrize("shift", [0, 1, 2])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_direct_force_matches_the_oracle(wm, oracle_mod, nx, shift, dtype):
    case = inputs.flat((nx, 7, 9), wall_height=-1.0, lengths=(2.0, 1.0, 1.0), sigma=0.1, seed=4)
    h = wm.Handle.from_case(case, dtype=dtype)
    h.set_tuning(force_path=2)
    tau = [_shifted(to_dev(case.tau[k], dtype), shift) for k in inputs.TAU_NAMES]
    f = [_shifted(torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda"), shift) for _ in range(3)]
    h.force(tau, f)
    ref = oracle_mod.force(case.grid, {k: to_host(to_dev(case.tau[k], dtype)) for k in inputs.TAU_NAMES})
    for got, want in zip(f, ref):
        got = to_host(got)
        assert np.all(np.isfinite(got))
        assert normwise(got, want)[0] <= TOL[dtype]


@pytest.mark.parametrize("shape,height", [((8, 4, 6), 0.4), ((64, 32, 12), 0.4), ((96, 80, 12), 0.4),
                                          ((160, 128, 10), 0.5), ((32, 16, 12), -1.0), ((32, 16, 12), 3.0)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_wall_stress_of_bands_of_all_sizes(wm, oracle_mod, shape, height, dtype):
    case = inputs.flat(shape, wall_height=height, sigma=0.1, seed=6)
    h = wm.Handle.from_case(case, dtype=dtype)
    rd = lambda a: to_host(to_dev(a, dtype))
    tau = [to_dev(case.tau[k], dtype) for k in inputs.TAU_NAMES]
    stats = h.new_stats()
    h.wall_stress(*[to_dev(x, dtype) for x in (case.u, case.v, case.w)], tau, stats)
    ref = {k: rd(case.tau[k]) for k in inputs.TAU_NAMES}
    ostats = oracle_mod.wall_stress(case.grid, case.phi_uv, case.phi_w, case.z0, case.phi_c, case.phi_b, rd(case.u),
                                    rd(case.v), rd(case.w), ref)
    for k, t in zip(inputs.TAU_NAMES, tau):
        assert normwise(to_host(t), ref[k])[0] <= TOL[dtype], k
    st = h.parse_stats(stats)
    for b in range(2):
        assert int(st[b]["count"]) == int(ostats[b, 0])
        assert abs(float(st[b]["sum_tw"]) - ostats[b, 1]) <= TOL[dtype] * max(abs(ostats[b, 1]), 1e-300) * 10
