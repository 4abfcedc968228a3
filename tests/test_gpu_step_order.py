"""A step sees what came before it in stream order although its wall kernel is placed
early: steps back to back, in-stream copies, copies from pinned memory and writes on
another stream joined by an event, each without a host synchronisation, bit for bit
the steps with a synchronisation on either side."""
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


CASES = {"cubes": lambda: inputs.cubes(shape=(128, 64, 64)), "ragged": lambda: inputs.hill(shape=(99, 61, 40)),
         "small": lambda: inputs.hill(shape=(32, 32, 16))}


def _set(case, dtype, vel, scale):
    vdt = torch.bfloat16 if vel == "bf16" else None
    uvw = [(scale * to_dev(x, dtype)).to(vdt) if vdt else scale * to_dev(x, dtype) for x in (case.u, case.v, case.w)]
    return uvw, [scale * to_dev(case.tau[k], dtype) for k in inputs.TAU_NAMES]


@pytest.mark.parametrize("own_stream", [False, True])
@pytest.mark.parametrize("dtype,vel", [("f32", "f32"), ("f32", "bf16"), ("f64", "f64")])
@pytest.mark.parametrize("name", sorted(CASES))
def test_steps_follow_the_stream(wm, name, dtype, vel, own_stream):
    case = CASES[name]()
    h = wm.Handle.from_case(case, dtype=dtype, vel_dtype=vel)
    sets = [_set(case, dtype, vel, s) for s in (1.0, -0.5, 0.25)]
    pinned = [([x.cpu().pin_memory() for x in u], [x.cpu().pin_memory() for x in t]) for u, t in sets]
    work = [x.clone() for x in sets[0][0]], [x.clone() for x in sets[0][1]]
    f = [torch.empty(h.shape, dtype=h.torch_dtype, device="cuda") for _ in range(3)]
    main = torch.cuda.Stream() if own_stream else torch.cuda.current_stream()
    side = torch.cuda.Stream()
    torch.cuda.synchronize()

    def load(src, how):
        if how == "side":
            side.wait_stream(main)
            with torch.cuda.stream(side):
                torch.cuda._sleep(20000)
                for d, x in zip(work[0] + work[1], src[0] + src[1]):
                    d.copy_(x)
            main.wait_stream(side)
        else:
            for d, x in zip(work[0] + work[1], src[0] + src[1]):
                d.copy_(x, non_blocking=True)

    def step(sync):
        if sync:
            torch.cuda.synchronize()
        h.step(*work[0], work[1], f)
        if sync:
            torch.cuda.synchronize()
        return [x.clone() for x in f + work[0] + work[1]]

    with torch.cuda.stream(main):
        ref = []
        for src in sets:
            load(src, "device")
            ref.append([step(True) for _ in range(3)])
        got = []
        for how in ("device", "side", "pinned"):
            for n in range(12):
                s = n % len(sets)
                load((pinned if how == "pinned" else sets)[s], how)
                got.append((s, [step(False) for _ in range(3)]))
        load(sets[1], "device")
        for _ in range(40):             # nothing between the steps
            h.step(*work[0], work[1], f)
        back = [x.clone() for x in f + work[0] + work[1]]
        load(sets[1], "device")
        for _ in range(40):
            torch.cuda.synchronize()
            h.step(*work[0], work[1], f)
        torch.cuda.synchronize()
    for s, outs in got:
        for a, b in zip(outs, ref[s]):
            assert all(torch.equal(x, y) for x, y in zip(a, b))
    assert all(torch.equal(x, y) for x, y in zip(back, f + work[0] + work[1]))
    assert h.device_status() == wm.OK
