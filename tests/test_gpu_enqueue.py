"""A step only enqueues, whichever way it is launched."""
import pytest

import paper_2409_04521_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu


def test_a_step_does_not_wait_for_the_gpu():
    torch = pytest.importorskip("torch")
    p = W.cosmo16(n=16, nsteps=12, nsrc=4, seed=4)
    stream = torch.cuda.Stream()
    s = F.Simulation(p, ray_capacity=1 << 20, stream=stream.cuda_stream)
    waited = []
    for k in range(26):
        if k == 13:
            s.set_launch(0, 2, 0, 128, 64)                # another launch: direct steps, then a new graph
        stream.synchronize()
        done = torch.cuda.Event()
        with torch.cuda.stream(stream):
            torch.cuda._sleep(100_000_000)                # some 50 ms, many times what a step's host work takes
            done.record()
        s.step(p.dt)
        if done.query():
            waited.append(k)
    assert waited == []
    s.close()
