"""The adjoint's transpose map built in windows of the grid, as on a device without room
for all of it (the injected failure of the map's first allocation; the windows begin and
end inside both grids' slots): the gradients bit for bit those with the map built at once."""
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


@pytest.mark.parametrize("dtype", ["f32", "f64"])
def test_map_in_windows(wm, monkeypatch, dtype):
    case, g = inputs.adjoint_case(shape=(120, 110, 100), dtype=dtype)       # 646 chunks of slots: windows of 256
    s = to_dev(np.log(case.z0), dtype)
    uvw = [to_dev(x, dtype) for x in (case.u, case.v, case.w)]
    g = [to_dev(x, dtype) for x in g]

    def gradients(h):
        h.set_log_z0(s)
        out = [torch.full(h.shape, float("nan"), dtype=h.torch_dtype, device="cuda") for _ in range(4)]
        h.backward(g, uvw, *out)
        torch.cuda.synchronize()
        h.close()
        return out

    ref = gradients(wm.Handle.from_case(case, dtype=dtype))
    for k in range(1, 80):              # the smallest k with which init goes through fails the map's first allocation
        monkeypatch.setenv("WMIBM_FAULT", f"alloc:{k}")
        try:
            h = wm.Handle.from_case(case, dtype=dtype)
        except wm.WmibmError:
            continue
        break
    got = gradients(h)
    assert all(torch.equal(a, b) for a, b in zip(got, ref))
