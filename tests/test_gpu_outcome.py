"""A failed step's error is reported by every later step and sync, however
often and in whatever order they are called, until a reset or a checkpoint
load starts the run anew; what it starts is not reported as failed."""
import pytest

import paper_2409_04521_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu


def _fails(call):
    with pytest.raises(F.FlexRTError) as e:
        call()
    assert e.value.status == 3                            # FLEXRT_E_CAPACITY


@pytest.mark.parametrize("anew", ["reset", "load"])
@pytest.mark.parametrize("first", ["sync", "step"])
def test_an_error_stays_until_the_run_starts_anew(first, anew):
    p = W.cosmo16(n=24, nsteps=20, nsrc=5, seed=4)
    s = F.Simulation(p, ray_capacity=1 << 13)             # overflows within the run
    for _ in range(3):
        s.step(p.dt)
    blob, steps = s.save_state(), 3
    for _ in range(2):
        if first == "sync":
            try:
                for _ in range(p.nsteps):
                    s.step(p.dt)
            except F.FlexRTError:
                pass
            _fails(s.sync)
        else:
            s.fields(("T",))                              # a getter sees steps end without reporting them
            _fails(lambda: [(s.step(p.dt), s.fields(("T",))) for _ in range(p.nsteps)])
        for _ in range(3):
            _fails(s.sync)
            _fails(lambda: s.step(p.dt))
            _fails(s.save_state)
        if anew == "reset":
            s.reset()
            steps = 0
        else:
            s.load_state(blob)
        s.sync()
        s.step(p.dt)
        s.sync()
        assert s.counts()["step"] == steps + 1
    s.close()
