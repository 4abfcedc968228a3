"""wmibm_wall_stress_force_from: the forcing bit for bit that of wmibm_wall_stress_force
on a copy of the stresses, which stay as they are, where the pipelined stencil reads
clean levels from the caller (band anywhere in the grid, at the floor, none at all)
and where it does not take the grid (rows that no vector divides, misaligned
stresses); a work buffer that is too small is refused."""
import ctypes

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


def _flat(shape, height):
    return inputs.flat(shape, wall_height=height, sigma=0.1, seed=2)


CASES = {"hill": lambda: inputs.hill(shape=(64, 32, 40)), "cubes": lambda: inputs.cubes(shape=(96, 48, 40)),
         "ragged": lambda: inputs.hill(shape=(63, 20, 17)), "no band": lambda: _flat((32, 16, 12), -1.0),
         "floor": lambda: _flat((32, 16, 12), 0.0), "middle": lambda: _flat((32, 16, 24), 0.5),
         "under the lid": lambda: _flat((32, 16, 24), 0.93), "all solid": lambda: _flat((32, 16, 12), 3.0)}


def _fields(wm, case, dtype, shift=0):
    h = wm.Handle.from_case(case, dtype=dtype)
    vel = [to_dev(x, dtype) for x in (case.u, case.v, case.w)]
    tau = []
    for k in inputs.TAU_NAMES:
        t = to_dev(case.tau[k], dtype)
        buf = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)
        tau.append(buf[shift:].view(t.shape).copy_(t))
    f = [[torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda") for _ in range(3)] for _ in range(2)]
    return h, vel, tau, f


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("shift", [0, 1])
@pytest.mark.parametrize("name", sorted(CASES))
def test_equals_the_stage_on_a_copy(wm, name, shift, dtype):
    case = CASES[name]()
    h, vel, tau, (f, ref) = _fields(wm, case, dtype, shift)
    before = [t.clone() for t in tau]
    copy = [t.clone() for t in tau]
    stats, stats_ref = h.new_stats(), h.new_stats()
    h.wall_stress_force(*vel, copy, ref, stats_ref)
    h.wall_stress_force_from(*vel, tau, f, stats)
    torch.cuda.synchronize()
    assert all(torch.equal(a, b) for a, b in zip(tau, before))
    assert all(torch.equal(a, b) for a, b in zip(f, ref))
    a, b = h.parse_stats(stats), h.parse_stats(stats_ref)
    assert np.array_equal(a["count"], b["count"]) and np.array_equal(a["min_tw"], b["min_tw"])
    assert h.device_status() == wm.OK


def test_a_small_work_buffer_is_refused(wm):
    h, vel, tau, (f, _) = _fields(wm, CASES["hill"](), "f32")
    ptrs = (ctypes.c_void_p * 6)(*[t.data_ptr() for t in tau])
    fp = [t.data_ptr() for t in f]
    need = h._L.wmibm_stage_work_bytes(h.raw, ptrs, *fp)
    assert 0 < need < 6 * tau[0].numel() * 4
    work = torch.empty(need, dtype=torch.uint8, device="cuda")
    st = h._L.wmibm_wall_stress_force_from(h.raw, *[t.data_ptr() for t in vel], ptrs, work.data_ptr(), need - 1, *fp,
                                           None, None)
    assert st == wm.EINVAL
    assert h._L.wmibm_stage_work_bytes(h.raw, ptrs, None, fp[1], fp[2]) == -1
