"""Steps with nothing between them, each with values of its own: every forcing, and the
stresses and velocities at the end, bit for bit those of the same steps with a
synchronisation after each.  Two steps in a row share a velocity, which the first one's
mask changes (by its own pressure gradient) before the second one's wall model gathers
it, and all steps share the stress arrays, whose wall values each one writes anew.
Planes of whole 32-byte sectors and others."""
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


# on the first three, some band node's gather meets a masked node
CASES = {"cubes": lambda: inputs.cubes(shape=(128, 64, 64)), "half sectors": lambda: inputs.cubes(shape=(44, 23, 24)),
         "ragged": lambda: inputs.cubes(shape=(127, 63, 62)), "hill": lambda: inputs.hill(shape=(256, 128, 48))}
PAIRS = 5


@pytest.mark.parametrize("dtype,vel", [("f32", "f32"), ("f32", "bf16"), ("f64", "f64")])
@pytest.mark.parametrize("name", sorted(CASES))
def test_back_to_back_steps_with_changing_values(wm, name, dtype, vel):
    case = CASES[name]()
    h = wm.Handle.from_case(case, dtype=dtype, vel_dtype=vel)
    vdt = torch.bfloat16 if vel == "bf16" else h.torch_dtype
    uvw = [to_dev(x, dtype) for x in (case.u, case.v, case.w)]
    tau0 = [to_dev(case.tau[k], dtype) for k in inputs.TAU_NAMES]
    # scales and pressure gradients (up to a few times the velocity, after the factor dt) of each pair of steps
    vels = [[((1.0 - 0.3 * n) * x).to(vdt) for x in uvw] for n in range(PAIRS)]
    grads = [[(0.5 + 0.7 * n) * x for x in reversed(uvw)] for n in range(2 * PAIRS)]

    def run(sync):
        tau, state = [t.clone() for t in tau0], [[x.clone() for x in s] for s in vels]
        f = [[torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda") for _ in range(3)]
             for _ in grads]
        torch.cuda.synchronize()
        for n, g in enumerate(grads):
            h.step(*state[n // 2], tau, f[n], g, 1.0)
            if sync:
                torch.cuda.synchronize()
        torch.cuda.synchronize()
        return f, [tau] + state

    f_ref, end_ref = run(True)
    if name != "hill":          # the second step of a pair gathers what the first one's mask left
        assert all(not torch.equal(f_ref[2 * n][0], f_ref[2 * n + 1][0]) for n in range(PAIRS))
    for _ in range(4):
        f, end = run(False)
        for a, b in zip(f + end, f_ref + end_ref):
            assert all(torch.equal(x, y) for x, y in zip(a, b))
    assert h.device_status() == wm.OK
