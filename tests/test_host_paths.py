"""The library's host code on a machine without a GPU: its objects are linked with a stand-in for the
CUDA runtime (fake_cudart.cpp) that keeps "device" memory on the host and records launches instead
of running them, so that failures can be made to happen (an allocation that does not succeed, a
device that stops answering) and the host's own decisions can be read off."""
import ctypes
import glob
import os
import subprocess

import numpy as np
import pytest

from paper_1302_5010_gb300 import build as libbuild
from paper_1302_5010_gb300 import mpl

HERE = os.path.dirname(os.path.abspath(__file__))
REGS = 96  # registers a thread of the split TF32 kernel is compiled to


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    libbuild.build()
    tmp = tmp_path_factory.mktemp("fake")
    obj, out = str(tmp / "fake.o"), str(tmp / "libmpl_host.so")
    cuda = os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(libbuild.nvcc()))), "include")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-w", "-I", libbuild.INCLUDE, "-I", cuda, "-c",
                    os.path.join(HERE, "fake_cudart.cpp"), "-o", obj], check=True, capture_output=True)
    objs = [os.path.join(libbuild.BUILD, os.path.basename(s)[:-3] + ".o") for s in libbuild._sources()]
    subprocess.run(["g++", "-shared", "-o", out, obj, *objs, "-Wl,-Bsymbolic", "-Wl,-z,defs", "-lpthread"], check=True,
                   capture_output=True)
    h = ctypes.CDLL(out)
    h.mpl_set_option.argtypes = [ctypes.c_void_p, ctypes.c_int, ctypes.c_double]
    for f in ("mpl_create", "bmpl_solve", "mpl_correlate", "mpl_correlate_noalloc", "mpl_proposal_set_weights",
              "mpl_proposal_loss_grad", "mpl_autotune"):
        getattr(h, f).restype = ctypes.c_int
    h.fake_set.argtypes = [ctypes.c_int] * 5 + [ctypes.c_uint]
    return h


def fake(lib, regs=REGS, fail_malloc=0, iterations=1, delay_us=0, view_on=1, flags=0):
    lib.fake_set(regs, fail_malloc, iterations, delay_us, view_on, flags)


def _f32(a):
    return a.ctypes.data_as(ctypes.c_void_p)


class Handle:
    def __init__(self, lib, n, m, **opts):
        self.lib, self.n, self.m = lib, n, m
        self.h = ctypes.c_void_p()
        A = np.zeros((m, n), dtype=np.float32)
        assert lib.mpl_create(_f32(A), n, m, ctypes.byref(self.h)) == mpl.MPL_OK
        for k, v in opts.items():
            assert lib.mpl_set_option(self.h, getattr(mpl, "MPL_OPT_" + k), float(v)) == mpl.MPL_OK

    def solve(self, p):
        B, lam = np.ones((p, self.n), dtype=np.float32), np.ones(p, dtype=np.float32)
        X = np.zeros((p, self.m), dtype=np.float32)
        return self.lib.bmpl_solve(self.h, _f32(B), p, _f32(lam), _f32(X), ctypes.c_double(1e-6), None)

    def close(self):
        self.lib.mpl_destroy(self.h)


def test_the_stand_in_runs_a_solve(lib):
    fake(lib, iterations=3)
    s = Handle(lib, 128, 300, RHO=2)
    assert s.solve(5) == mpl.MPL_OK
    assert lib.fake_count(b"cudaGraphLaunch") == 3
    s.close()
    assert lib.fake_live() == 0


@pytest.mark.parametrize("graph", [0, 1])
def test_a_solve_that_fails_leaves_nothing_running(lib, graph):
    """A solve that returns an error half way has waited for what it launched: its kernels use the
    handle's workspace, which the next call on the handle (any of them) uses as well."""
    s = Handle(lib, 128, 300, RHO=2, GRAPH=graph)
    fake(lib, view_on=0)  # the stream runs dry without the selection's results
    assert s.solve(5) == mpl.MPL_ERR_CUDA
    last = max(lib.fake_last(b"k_"), lib.fake_last(b"cudaGraphLaunch"))
    assert 0 <= last < lib.fake_last(b"cudaDeviceSynchronize")
    fake(lib)
    assert s.solve(5) == mpl.MPL_OK
    assert lib.fake_count(b"cudaDeviceSynchronize") == 0  # (and a sound one waits for its own stream only)
    s.close()


@pytest.mark.parametrize("k", range(1, 9))
def test_proposal_buffers_all_or_none(lib, k):
    """An allocation of the proposal network's buffers that fails leaves none of them behind: the next
    call makes them all, and the training pass has the rows it writes its sums to."""
    s = Handle(lib, 128, 300, RHO=2)
    w = np.zeros(mpl.MPL_PROPOSAL_NPARAM, dtype=np.float32)
    before = lib.fake_live()
    fake(lib, fail_malloc=k)
    assert lib.mpl_proposal_set_weights(s.h, _f32(w), w.size) == mpl.MPL_ERR_OOM
    assert lib.fake_live() == before
    assert lib.fake_count(b"k_sketch") == 0
    fake(lib)
    assert lib.mpl_proposal_set_weights(s.h, _f32(w), w.size) == mpl.MPL_OK
    B, lam = np.ones((3, 128), dtype=np.float32), np.ones(3, dtype=np.float32)
    X = np.zeros((3, 300), dtype=np.float32)
    loss, g = ctypes.c_double(), np.zeros_like(w)
    assert lib.mpl_proposal_loss_grad(s.h, _f32(B), 3, _f32(lam), _f32(X), ctypes.byref(loss), _f32(g)) == mpl.MPL_OK
    assert lib.fake_count(b"k_train_fwd_bwd") == 1 and not lib.fake_train_part_null()
    s.close()
    assert lib.fake_live() == 0


@pytest.mark.parametrize("p", [9, 300])
def test_correlation_without_the_registers_it_hands_out(lib, p):
    """The split TF32 kernel hands its loaders' registers to the warps that accumulate; compiled to too few it
    is not launched, and the FP32 chain, which computes the same product, takes the call."""
    n, m = 256, 300
    A, R, C = (np.zeros(s, dtype=np.float32) for s in ((m, n), (p, n), (p, m)))

    def aligned(a):
        b = np.zeros(a.size + 4, dtype=np.float32)
        return b[(-b.ctypes.data // 4) % 4:][:a.size]

    A, R, C = aligned(A), aligned(R), aligned(C)
    for regs, kernel in ((REGS, b"k_corr_tf32"), (94, b"k_corr_f32")):
        fake(lib, regs=regs)
        assert lib.mpl_correlate_noalloc(_f32(A), n, m, _f32(R), p, _f32(C), None) == mpl.MPL_OK
        assert lib.fake_count(b"k_corr_") == lib.fake_count(kernel) == 1


@pytest.mark.parametrize("n,p,tf32", [(64, 5, False), (64, 20, False), (128, 5, False), (200, 300, False),
                                      (255, 20, False), (256, 20, True), (256, 8, False), (256, 9, True),
                                      (400, 300, True), (1024, 5, False), (1024, 20, True)])
def test_band_of_the_kernels_that_run(lib, n, p, tf32):
    """The selection's error bound is that of the correlation kernels the batch can take: gamma_n for the
    chain (n < 256) and the matrix-vector products (at most 8 signals, n >= 256), the wider of
    that and the split TF32 form for the others.  (u = 2^-24; 2 gamma_n + rounding of the residual.)"""
    fake(lib)
    s = Handle(lib, n, 300, RHO=2)
    assert s.solve(p) == mpl.MPL_OK
    got = (ctypes.c_float * 5)()
    assert lib.fake_bounds(b"k_select", got) == 1
    s.close()
    u = 2.0 ** -24
    gam = n * u / (1 - n * u)
    chain = 2 * (gam + u)
    split = 1.25 * (98 * 2.0 ** -22 + (n / 32 + 2) * u)
    want = max(chain, split) if tf32 else chain
    np.testing.assert_allclose(got[:2], [want * 1.01] * 2, rtol=1e-6)
    assert got[3] == pytest.approx(chain * 1.01, rel=1e-6)
    assert got[4] == (np.float32(np.sqrt(n) * 2.0 ** -136) if tf32 else 0.0)
    smax = min(n, 256)
    gs = (smax + 1) * u / (1 - (smax + 1) * u)
    gb = max(gam, split) if tf32 else gam
    assert got[2] == pytest.approx((gb + 2 * gs * (1 + gb) + u) * 1.01, rel=1e-6)


@pytest.mark.parametrize("sync_every", [1, 2, 7])
def test_autotuner_times_each_setting_once(lib, sync_every):
    """MPL_OPT_SYNC_EVERY has no effect on a solve, so the tuner does not time its values against each other:
    one solve to warm up and three timed for each of four route lengths and, with the best of them, the
    gathered Gram rows.  The handle keeps the value it had."""
    s = Handle(lib, 128, 300, RHO=2, SYNC_EVERY=sync_every)
    p = 5
    B, lam = np.ones((p, 128), dtype=np.float32), np.ones(p, dtype=np.float32)
    out = mpl.TuneResult()
    fake(lib)
    assert lib.mpl_autotune(s.h, _f32(B), p, _f32(lam), ctypes.c_double(1e-6), None, ctypes.byref(out)) == mpl.MPL_OK
    assert lib.fake_count(b"6k_init") == 4 * (4 + 1)
    assert out.sync_every == sync_every and out.candidates == 3 * (4 + 1)
    v = ctypes.c_double()
    assert lib.mpl_get_option(s.h, mpl.MPL_OPT_SYNC_EVERY, ctypes.byref(v)) == mpl.MPL_OK and v.value == sync_every
    s.close()


@pytest.mark.parametrize("flag", [0, 1, 4])
def test_the_wait_for_the_work_lists_keeps_the_schedule_flag(lib, flag):
    """A process that asked for blocking synchronisation (cudaDeviceScheduleBlockingSync = 4) does not
    find a core polled at full rate while a solve runs: 10 iterations of 20 ms cost it a small part of
    200 ms.  Spinning (1) and no choice (0) only have to finish."""
    import time
    s = Handle(lib, 128, 300, RHO=2)
    fake(lib, iterations=1, flags=flag)
    assert s.solve(5) == mpl.MPL_OK
    fake(lib, iterations=10, delay_us=20000, flags=flag)
    w, c = time.perf_counter(), time.process_time()
    assert s.solve(5) == mpl.MPL_OK
    w, c = time.perf_counter() - w, time.process_time() - c
    s.close()
    assert w >= 0.2
    assert flag != 4 or c <= 0.5 * w, (w, c)


def test_the_wait_yields_where_asked(lib):
    """cudaDeviceScheduleYield (2): two solves in two threads still finish, and so does one whose device
    stops answering."""
    import threading
    fake(lib, iterations=20, delay_us=200, flags=2)
    rc = []

    def one():
        s = Handle(lib, 128, 300, RHO=2)
        rc.append(s.solve(5))
        s.close()

    ts = [threading.Thread(target=one) for _ in range(2)]
    for t in ts:
        t.start()
    for t in ts:
        t.join()
    assert rc == [mpl.MPL_OK] * 2
    for flag in (2, 4):
        fake(lib, view_on=0, flags=flag)
        s = Handle(lib, 128, 300, RHO=2)
        assert s.solve(5) == mpl.MPL_ERR_CUDA
        s.close()


@pytest.mark.parametrize("smax,waits", [(128, (1, 1, 1)), (4, (1, 2, 3))])
def test_profiling_leaves_the_iterations_overlapped(lib, smax, waits):
    """With MPL_OPT_PROFILE a replayed iteration's timing events are read when its graph is replayed again
    (iterations beyond the one where the active-set bound saturates share a graph per list slot:
    with smax 4 and rho 2 those of t = 8..11 repeat 4..7), or at the end: the host does not wait for an
    iteration before it queues the next.  Every iteration's phases are counted once."""
    s = Handle(lib, 128, 300, RHO=2, SMAX=smax, PROFILE=1)
    elapsed, waited = [], []
    for it in (6, 11, 16):
        fake(lib, iterations=it)
        assert s.solve(5) == mpl.MPL_OK
        assert lib.fake_count(b"cudaGraphLaunch") == it
        elapsed.append(lib.fake_count(b"cudaEventElapsedTime"))
        waited.append(lib.fake_count(b"cudaStreamSynchronize"))
    s.close()
    assert elapsed[1] - elapsed[0] == elapsed[2] - elapsed[1] > 0
    assert tuple(waited) == waits
