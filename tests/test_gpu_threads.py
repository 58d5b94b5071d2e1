"""Single simulations in host threads of their own, each making and remaking
its step's graph: on streams that wait for the legacy stream, beside threads
that wait for the whole device, and beside a capture of somebody else's."""
import ctypes
import threading

import numpy as np
import pytest

import paper_2409_04521_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu


def _prob():
    return W.cosmo16(n=16, nsteps=11, nsrc=4, seed=4)


def _blocking_streams(n):
    cu = ctypes.CDLL("libcuda.so.1")
    out = []
    for _ in range(n):
        h = ctypes.c_void_p()
        assert cu.cuStreamCreate(ctypes.byref(h), 0) == 0      # CU_STREAM_DEFAULT
        out.append(h.value)
    return cu, out


def _rounds(s, p, n, errors, waits):
    try:
        for k in range(n):
            s.set_launch(0, 2 + k % 2)                     # the graph is made again in every round
            s.reset()
            for i in range(p.nsteps):
                s.step(p.dt)
                if waits:
                    s.counts()
            s.sync()
    except Exception as e:                                 # noqa: BLE001 -- reported by the test's thread
        errors.append(repr(e))


def _beside(fn, n):
    th = [threading.Thread(target=fn, args=(k,)) for k in range(n)]
    for t in th:
        t.start()
    for t in th:
        t.join()


def _same(sims, p):
    ref = F.Simulation(p, ray_capacity=1 << 20)
    for _ in range(p.nsteps):
        ref.step(p.dt)
    for s in sims:
        assert s.counts() == ref.counts()
        # two runs differ by the order of their deposits: a few 1e-7 a step
        a, b = s.fields()["gamma_HI"], ref.fields()["gamma_HI"]
        assert np.allclose(a, b, rtol=1e-5, atol=1e-5 * b.max())
        s.close()
    ref.close()


def test_blocking_streams_in_threads():
    p = _prob()
    ref = F.Simulation(p, ray_capacity=1 << 20)            # (makes the primary context)
    cu, streams = _blocking_streams(3)
    sims = [F.Simulation(p, ray_capacity=1 << 20, stream=h) for h in streams]
    for s in sims:
        s.step(p.dt)
    errors = []
    _beside(lambda k: _rounds(sims[k], p, 60, errors, True), 3)
    assert errors == []
    _same(sims, p)
    ref.close()
    for h in streams:
        assert cu.cuStreamDestroy_v2(ctypes.c_void_p(h)) == 0


def test_threads_that_wait_for_the_device():
    torch = pytest.importorskip("torch")
    p = _prob()
    sims = [F.Simulation(p, ray_capacity=1 << 20) for _ in range(2)]
    errors, done = [], threading.Event()

    def waiter():
        try:
            while not done.is_set():
                torch.cuda.synchronize()
        except Exception as e:                             # noqa: BLE001
            errors.append(repr(e))

    w = threading.Thread(target=waiter)
    w.start()
    _beside(lambda k: _rounds(sims[k], p, 100, errors, False), 2)
    done.set()
    w.join()
    assert errors == []
    _same(sims, p)


def test_beside_a_capture_of_another_thread():
    torch = pytest.importorskip("torch")
    p = _prob()
    s = F.Simulation(p, ray_capacity=1 << 20)
    s.step(p.dt)
    s.sync()
    errors = []

    def rest():
        try:
            for _ in range(p.nsteps - 1):                  # past the step that makes the graph
                s.step(p.dt)
        except Exception as e:                             # noqa: BLE001
            errors.append(repr(e))

    x = torch.zeros(8, device="cuda")
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g):                              # other threads' unsafe calls would end it
        x += 1
        t = threading.Thread(target=rest)
        t.start()
        t.join()
        x += 1
    g.replay()
    torch.cuda.synchronize()
    assert errors == [] and x.tolist() == [2.0] * 8
    _same([s], p)
