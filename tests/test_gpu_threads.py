"""Two host threads, each with a grid, a handle and a stream of its own, calling a kernel
whose shared memory depends on the grid: no call fails, and each result is that of the
thread alone, bit for bit.  The threads are C++ ones, so that their calls overlap."""
import ctypes
import os
import subprocess

import pytest

from paper_2006_03343_gb300 import inputs

from parity_util import to_dev

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

CALLS = 3000
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SOURCE = r"""
#include <atomic>
#include <thread>
#include "wmibm.h"
struct Job {
    wmibm_handle *h;
    const void *vel[3], *wt[2];
    void *tau[6], *f[3], *stream;
};
// failed calls of two threads that call entry `what` n times each
extern "C" int run(int what, void *entry, const Job *jobs, int n)
{
    std::atomic<int> ready{0}, failed{0};
    auto loop = [&](const Job &j) {
        for (++ready; ready < 2;) {}
        for (int i = 0; i < n; ++i) {
            int st = 0;
            if (what == 0)
                st = ((decltype(&wmibm_sgs_stress))entry)(j.h, j.vel[0], j.vel[1], j.vel[2], j.wt[0], j.wt[1], j.tau, 0.16,
                                                          j.stream);
            else if (what == 1)
                st = ((decltype(&wmibm_sgs_force))entry)(j.h, j.vel[0], j.vel[1], j.vel[2], j.wt[0], j.wt[1],
                                                         (const void *const *)j.tau, j.f[0], j.f[1], j.f[2], 0.16, j.stream);
            else
                st = ((decltype(&wmibm_force_spectral))entry)(j.h, (const void *const *)j.tau, j.f[0], j.f[1], j.f[2],
                                                              j.stream);
            if (st) ++failed;
        }
    };
    std::thread a(loop, jobs[0]), b(loop, jobs[1]);
    a.join();
    b.join();
    return failed;
}
"""


class Job(ctypes.Structure):
    _fields_ = [("h", ctypes.c_void_p), ("vel", ctypes.c_void_p * 3), ("wt", ctypes.c_void_p * 2),
                ("tau", ctypes.c_void_p * 6), ("f", ctypes.c_void_p * 3), ("stream", ctypes.c_void_p)]


@pytest.fixture(scope="module")
def wm():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2006_03343_gb300 import build, wmibm
    build.build()
    wmibm.load()
    return wmibm


@pytest.fixture(scope="module")
def threads(tmp_path_factory):
    d = tmp_path_factory.mktemp("threads")
    (d / "threads.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-std=c++17", "-shared", "-fPIC", "-pthread", f"-I{ROOT}/include",
                    str(d / "threads.cpp"), "-o", str(d / "threads.so")], check=True)
    return ctypes.CDLL(str(d / "threads.so"))


ENTRIES = ["sgs_stress", "sgs_force", "force_spectral"]


@pytest.mark.parametrize("dtype", ["f32", "f64"])
@pytest.mark.parametrize("what", ENTRIES)
def test_two_threads_with_two_grids(wm, threads, what, dtype):
    jobs, results, keep = (Job * 2)(), [], []
    for job, shape in zip(jobs, ((16, 8, 8), (256, 64, 8))):
        case = inputs.hill(shape=shape)
        h = wm.Handle.from_case(case, dtype=dtype)
        vel = [to_dev(x, dtype) for x in (case.u, case.v, case.w)]
        tau = [to_dev(case.tau[k], dtype) for k in inputs.TAU_NAMES]
        f = [torch.zeros(h.shape, dtype=h.torch_dtype, device="cuda") for _ in range(3)]
        wt = h.sgs_wall_terms(case.phi_uv, case.phi_w, case.z0)
        if what == "sgs_stress":
            h.sgs_stress(*vel, wt, tau)
        elif what == "sgs_force":
            h.wall_stress(*vel, tau)
            h.sgs_force(*vel, wt, tau, f)
        else:
            h.force_spectral(tau, f)
        stream = torch.cuda.Stream()
        results.append((tau + f, [t.clone() for t in tau + f]))
        keep.append((h, vel, wt, stream))
        job.h, job.stream = h.raw, stream.cuda_stream
        for name, seq in (("vel", vel), ("wt", wt), ("tau", tau), ("f", f)):
            getattr(job, name)[:] = [t.data_ptr() for t in seq]
    torch.cuda.synchronize()
    entry = ctypes.cast(getattr(keep[0][0]._L, "wmibm_" + what), ctypes.c_void_p)
    code = ("sgs_stress", "sgs_force", "force_spectral").index(what)
    failed = threads.run(code, entry, jobs, CALLS)
    torch.cuda.synchronize()
    assert failed == 0
    for got, ref in results:
        assert all(torch.equal(a, b) for a, b in zip(got, ref))
    assert all(k[0].device_status() == wm.OK for k in keep)
