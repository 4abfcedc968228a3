"""A captured batch step follows fields that are set after the capture, also where their
addresses no longer (or only now) keep every 32-byte sector within one level: replays
bit for bit the members' separate calls."""
import pytest

from paper_2006_03343_gb300 import inputs

from parity_util import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

SHAPES = ((64, 32, 24), (48, 24, 16), (128, 16, 32))       # planes of whole sectors in both precisions


@pytest.fixture(scope="module")
def wm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_03343_gb300 import build, wmibm
    build.build()
    wmibm.load()
    return wmibm


def _moved(t, nbytes):
    n = nbytes // t.element_size()
    buf = torch.empty(t.numel() + n, dtype=t.dtype, device=t.device)
    return buf[n:].view(t.shape).copy_(t)


def _fields(h, case, dtype, scale, nbytes):
    uvw = [scale * to_dev(x, dtype) for x in (case.u, case.v, case.w)]
    tau = [_moved(scale * to_dev(case.tau[k], dtype), nbytes) for k in inputs.TAU_NAMES]
    f = [_moved(torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda"), nbytes) for _ in range(3)]
    return uvw, tau, f


@pytest.mark.parametrize("first,then", [(0, 16), (16, 0)])
@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_replay_with_other_addresses(wm, dtype, first, then):
    cases = [inputs.ensemble_member(m, shape=s, dtype=dtype) for m, s in enumerate(SHAPES)]
    handles = [wm.Handle.from_case(c, dtype=dtype) for c in cases]
    batch = wm.Batch(handles)

    def sets(scale, nbytes):
        return [_fields(h, c, dtype, scale, nbytes) for h, c in zip(handles, cases)]

    captured = sets(1.0, first)
    batch.set_fields([(*uvw, tau, f) for uvw, tau, f in captured])
    batch.step()
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        batch.step()
    got, ref = sets(-0.5, then), sets(-0.5, then)
    batch.set_fields([(*uvw, tau, f) for uvw, tau, f in got])
    for n in range(3):
        graph.replay()
        for h, (uvw, tau, f) in zip(handles, ref):
            h.wall_stress(*uvw, tau)
            h.force(tau, f)
            h.mask(*uvw)
        for a, b in zip(got, ref):
            assert all(torch.equal(x, y) for p, q in zip(a, b) for x, y in zip(p, q)), n
            for x, y in zip(a[0], b[0]):        # other velocities for the next replay
                assert x.data_ptr() != y.data_ptr()
                x.mul_(-0.75)
                y.mul_(-0.75)
    assert handles[0].device_status() == wm.OK
    batch.close()
