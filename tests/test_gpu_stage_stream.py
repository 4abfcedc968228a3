"""wmibm_wall_stress_force_from on a stream of the caller's while the current stream has
work pending."""
import ctypes

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


def test_work_buffer_belongs_to_the_given_stream(wm):
    """A block freed on the current stream while a kernel there still has to read it is
    not taken as the work buffer of a call on another stream."""
    case = inputs.hill(shape=(64, 32, 40))
    h = wm.Handle.from_case(case)
    vel = [to_dev(x, "f32") for x in (case.u, case.v, case.w)]
    tau = [to_dev(case.tau[k], "f32") for k in inputs.TAU_NAMES]
    f, ref = ([torch.empty(h.shape, dtype=torch.float32, device="cuda") for _ in range(3)] for _ in range(2))
    h.wall_stress_force_from(*vel, tau, ref)
    ptrs = (ctypes.c_void_p * 6)(*[t.data_ptr() for t in tau])
    need = h._L.wmibm_stage_work_bytes(h.raw, ptrs, *[t.data_ptr() for t in f])
    side = torch.cuda.Stream()
    block = torch.full((need,), 77, dtype=torch.uint8, device="cuda")
    seen = torch.empty_like(block)
    torch.cuda.synchronize()
    torch.cuda._sleep(20_000_000)               # some 10 ms; the copy below comes after it
    seen.copy_(block)
    del block
    h.wall_stress_force_from(*vel, tau, f, stream=side)
    torch.cuda.synchronize()
    assert bool((seen == 77).all())
    assert all(torch.equal(a, b) for a, b in zip(f, ref))
    assert h.device_status() == wm.OK
