"""Views as the given stresses of the differentiable stage: slices and expanded views give
the forcing of their dense copies, bit for bit, and stay as they are; a permuted view, whose
memory order is not the fields', is refused."""
import numpy as np
import pytest

from paper_2006_03343_gb300 import autograd, inputs

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


def _sliced(t):
    wide = torch.zeros(*t.shape[:2], 2 * t.shape[2], dtype=t.dtype, device=t.device)
    return wide[..., ::2].copy_(t)


def _expanded(t):
    return t[:1].expand(t.shape)


def _permuted(t):
    return t.permute(2, 1, 0).contiguous().permute(2, 1, 0)


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("view", [_sliced, _expanded, _permuted])
def test_views_of_the_given_stresses(wm, view, dtype):
    case = inputs.hill(shape=(48, 20, 24))
    h = wm.Handle.from_case(case, dtype=dtype)
    uvw = [to_dev(x, dtype) for x in (case.u, case.v, case.w)]
    s = to_dev(np.log(case.z0), dtype)
    views = [view(to_dev(case.tau[k], dtype)) for k in inputs.TAU_NAMES]
    assert not any(t.is_contiguous() for t in views)
    if view is _permuted:
        with pytest.raises(ValueError):
            autograd.wall_stress_force(h, *uvw, s, views)
        return
    dense = [t.contiguous() for t in views]
    before = [t.clone() for t in dense]
    ref = autograd.wall_stress_force(h, *uvw, s, dense)
    got = autograd.wall_stress_force(h, *uvw, s, views)
    assert all(torch.equal(a, b) for a, b in zip(got, ref))
    assert all(torch.equal(a, b) for a, b in zip(views, before))
