"""The untuned stage (the direct-load stencil dependent on the wall kernel, the body
mask in the same launch) bit for bit that of the separate calls, wall stress, force
and mask, and of the two-launch pipeline where its rows and addresses allow that one:
planes of whole 32-byte sectors and others, rows of four, two and single values,
misaligned fields, bands at the floor, inside, at the lid, everywhere and nowhere,
every velocity type; and batches of members that differ in all of this."""
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


SHAPES = [(32, 16, 20), (36, 5, 24), (132, 7, 31), (66, 10, 12), (63, 20, 17), (4, 3, 5), (260, 2, 9), (8, 33, 34)]
HEIGHTS = {"none": -1.0, "floor": 0.0, "middle": 0.5, "lid": 0.93, "solid": 3.0}


def _case(shape, height, seed=7):
    return inputs.flat(shape, wall_height=HEIGHTS[height], sigma=0.1, seed=seed, lengths=(2.0, 1.0, 1.0))


def _moved(t, shift):
    buf = torch.empty(t.numel() + shift, dtype=t.dtype, device=t.device)
    return buf[shift:].view(t.shape).copy_(t)


def _state(h, case, dtype, vel, shift):
    vdt = torch.bfloat16 if vel == "bf16" else h.torch_dtype
    uvw = [_moved(to_dev(x, dtype).to(vdt), shift) for x in (case.u, case.v, case.w)]
    tau = [_moved(to_dev(case.tau[k], dtype), shift) for k in inputs.TAU_NAMES]
    f = [_moved(torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda"), shift) for _ in range(3)]
    g = [_moved(to_dev(case.tau[k], dtype), shift) for k in inputs.TAU_NAMES[:3]]
    return uvw, tau, f, g


def _same(a, b):
    return all(torch.equal(x, y) for p, q in zip(a[:3], b[:3]) for x, y in zip(p, q))


@pytest.mark.parametrize("dtype,vel", [("f32", "f32"), ("f32", "bf16"), ("f64", "f64")])
@pytest.mark.parametrize("height", sorted(HEIGHTS))
@pytest.mark.parametrize("shape", SHAPES)
def test_untuned_stage_equals_the_separate_calls(wm, shape, height, dtype, vel):
    case = _case(shape, height)
    h = wm.Handle.from_case(case, dtype=dtype, vel_dtype=vel)
    pipe = wm.Handle.from_case(case, dtype=dtype, vel_dtype=vel)
    pipe.set_tuning(force_path=3)
    for shift in (0, 1):
        for dt in (0.0, 0.25):
            ref, got, two = (_state(h, case, dtype, vel, shift) for _ in range(3))
            stats = [h.new_stats() for _ in range(3)]
            h.wall_stress(*ref[0], ref[1], stats[0])
            h.force(ref[1], ref[2])
            h.mask(*ref[0], ref[3] if dt else None, dt)
            h.step(*got[0], got[1], got[2], got[3] if dt else None, dt, stats[1])
            pipe.step(*two[0], two[1], two[2], two[3] if dt else None, dt, stats[2])
            torch.cuda.synchronize()
            assert _same(got, ref) and _same(two, ref), (shift, dt)
            a, b, c = (h.parse_stats(s) for s in stats)
            for x in (b, c):
                assert np.array_equal(a["count"], x["count"]) and np.array_equal(a["min_tw"], x["min_tw"])
        got, split = (_state(h, case, dtype, vel, shift) for _ in range(2))
        h.wall_stress_force(*got[0], got[1], got[2])
        h.wall_stress(*split[0], split[1])
        h.force_mask(split[1], split[2], *split[0], split[3], 0.25)
        ref = _state(h, case, dtype, vel, shift)
        h.wall_stress(*ref[0], ref[1])
        h.force(ref[1], ref[2])
        assert all(torch.equal(x, y) for x, y in zip(got[1] + got[2], ref[1] + ref[2])), shift
        h.mask(*ref[0], ref[3], 0.25)
        assert _same(split, ref), shift
    assert h.device_status() == wm.OK


@pytest.mark.parametrize("dtype,vel", [("f32", "f32"), ("f32", "bf16"), ("f64", "f64")])
@pytest.mark.parametrize("count", [1, 8])
def test_untuned_batch_equals_the_separate_calls(wm, count, dtype, vel):
    shapes = [s for s in SHAPES if s[0] % 4 == 0 and s[1] >= 3]      # what a batch takes
    names = sorted(HEIGHTS)
    cases = [_case(shapes[m % len(shapes)], names[m % len(names)], seed=m) for m in range(count)]
    handles = [wm.Handle.from_case(c, dtype=dtype, vel_dtype=vel) for c in cases]
    got = [_state(h, c, dtype, vel, 0) for h, c in zip(handles, cases)]
    batch = wm.Batch(handles)
    batch.set_fields([(*s[0], s[1], s[2]) for s in got])
    batch.step()
    for h, c, s in zip(handles, cases, got):
        ref = _state(h, c, dtype, vel, 0)
        h.wall_stress(*ref[0], ref[1])
        h.force(ref[1], ref[2])
        h.mask(*ref[0])
        assert _same(s, ref), c.shape
    assert handles[0].device_status() == wm.OK
    batch.close()
