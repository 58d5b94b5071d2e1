"""Steps of a single simulation replayed from a graph: the same run as direct
launches, the same error behaviour, and a caller's own capture of a step."""
import dataclasses as dc

import numpy as np
import pytest

import paper_2409_04521_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu
# two runs differ by the order of their single-precision deposits: a few times
# 1e-7 a step in Gamma and the opacities, under 1e-5 over these runs
RTOL = 1e-5


def _prob(**kw):
    p = W.cosmo16(n=24, nsteps=20, nsrc=5, seed=4)
    return dc.replace(p, options=dc.replace(p.options, **kw))


def _same(a, b):
    for k in ("gamma_HI", "T", "x_HII"):
        assert np.allclose(a[k], b[k], rtol=RTOL, atol=RTOL * np.abs(b[k]).max()), k


# (Generalized mode runs replayed steps against the oracle in its own tests)
@pytest.mark.parametrize("kw", [{}, dict(gamma_iters=3)])
def test_replayed_steps_equal_direct_ones(kw):
    p = _prob(**kw)
    a, b = F.Simulation(p, ray_capacity=1 << 21), F.Simulation(p, ray_capacity=1 << 21)
    b.profile(True)                                       # profiled steps are launched directly
    for k in range(p.nsteps):
        if k == 14:
            a.set_launch(0, 2, 0, 128, 64)                # another launch: the graph is made again
        a.step(p.dt if k != 11 else 0.5 * p.dt)           # the step length is not part of the graph
        b.step(p.dt if k != 11 else 0.5 * p.dt)
    assert a.counts() == b.counts()
    _same(a.fields(), b.fields())
    a.close()
    b.close()


def test_overflow_in_a_replayed_step_keeps_the_last_state():
    p = _prob()
    ref = F.Simulation(p, ray_capacity=1 << 21)
    rays = []
    for _ in range(p.nsteps):
        ref.step(p.dt)
        rays.append(ref.counts()["rays"])
    cap = int(rays[12] / 1.25) - 4096                     # the queue holds 1.25 cap + 4096: step 13 or soon after
    s = F.Simulation(p, ray_capacity=cap)
    with pytest.raises(F.FlexRTError) as e:
        for _ in range(p.nsteps):
            s.step(p.dt)
        s.sync()
    assert e.value.status == 3
    n = s.counts()["step"]
    assert 8 < n < p.nsteps and s.counts()["rays"] == rays[n - 1]
    ref.reset()
    for _ in range(n):
        ref.step(p.dt)
    _same(s.fields(), ref.fields())
    s.reset()                                             # and the context works again
    for _ in range(n):
        s.step(p.dt)
    s.sync()
    _same(s.fields(), ref.fields())
    s.close()
    ref.close()


def test_a_callers_capture_of_a_step():
    torch = pytest.importorskip("torch")
    p = _prob()
    stream = torch.cuda.Stream()
    s = F.Simulation(p, ray_capacity=1 << 21, stream=stream.cuda_stream)
    ref = F.Simulation(p, ray_capacity=1 << 21)
    for _ in range(12):
        s.step(p.dt)
    s.sync()
    g = torch.cuda.CUDAGraph()
    with torch.cuda.graph(g, stream=stream):
        s.step(p.dt)
    with torch.cuda.stream(stream):
        for _ in range(3):
            g.replay()
    stream.synchronize()
    for _ in range(15):
        ref.step(p.dt)
    assert s.counts()["step"] == ref.counts()["step"] == 15
    _same(s.fields(), ref.fields())
    s.close()
    ref.close()
