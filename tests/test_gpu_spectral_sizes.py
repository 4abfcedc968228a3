"""The pseudo-spectral forcing on every power of two of a line, in x and in y, with
aligned fields (16-byte staging and epilogues) and with fields one value off a
16-byte boundary, against the FP64 oracle: 1e-5 of each array's largest value in
FP32, 1e-12 in FP64; both alignments agree bit for bit."""
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


def _moved(t, shift):
    buf = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)
    return buf[shift:].view(t.shape).copy_(t)


@pytest.mark.parametrize("dtype,log", [("f32", n) for n in range(1, 12)] + [("f64", n) for n in range(1, 11)])
def test_every_power_of_two(wm, oracle_mod, dtype, log):
    for shape in ((1 << log, 4, 4), (8, 1 << log, 3)):
        case = inputs.flat(shape, wall_height=0.1, lengths=(2 * np.pi, np.pi, 1.0))
        h = wm.Handle.from_case(case, dtype=dtype)
        rng = np.random.default_rng(log)
        src = {k: 0.1 * rng.standard_normal(shape[::-1]) for k in inputs.TAU_NAMES}
        out = []
        for shift in (0, 1):
            tau = [_moved(to_dev(src[k], dtype), shift) for k in inputs.TAU_NAMES]
            f = [_moved(torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda"), shift)
                 for _ in range(3)]
            h.force_spectral(tau, f)
            torch.cuda.synchronize()
            out.append(f)
        ref = oracle_mod.force_spectral(case.grid, {k: to_host(to_dev(src[k], dtype)) for k in inputs.TAU_NAMES})
        for got, off, want in zip(*out, ref):
            assert torch.equal(got, off)
            assert normwise(to_host(got), want)[0] <= TOL[dtype], shape
    assert h.device_status() == wm.OK
