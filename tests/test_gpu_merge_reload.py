"""A checkpoint loaded after a step that failed, inside the merge among other
places, is a fresh start: no photons of the failed step are left."""
import dataclasses as dc

import numpy as np
import pytest

import paper_2409_04521_gb300 as F
import workloads as W
from parity_util import BUDGET_RTOL

pytestmark = pytest.mark.gpu


def test_load_after_a_failure_inside_the_merge():
    p = W.cosmo16(n=32, nsteps=12, nsrc=600, seed=4)
    p = dc.replace(p, options=dc.replace(p.options, merge=True, n_ex=0.0, l_merge=0))
    ref = F.Simulation(p, ray_capacity=1 << 20)
    ref.step(p.dt)
    blob = ref.save_state()
    for _ in range(7):
        ref.step(p.dt)
    ref.step_stage(p.dt, 1)
    marched = len(ref.rays()["level"])
    ref.step_stage(p.dt, 2)
    left = ref.counts()["rays"]
    ref.close()
    assert 1 << 15 < marched and left < marched
    failed = 0
    # queues that hold the ninth march's output but only part of what its
    # merge appends (1.25 x the capacity + 4096 slots)
    for f in np.linspace(0.0, 1.0, 9):
        s = F.Simulation(p, ray_capacity=int((marched + f * left - 4096) / 1.25))
        try:
            for _ in range(p.nsteps):
                s.step(p.dt)
            s.sync()
        except F.FlexRTError:
            failed += 1
        s.load_state(blob)
        for _ in range(3):
            s.step(p.dt)
        b = s.budget()
        assert abs(b[0] - b[1] - b[2] - b[3]) <= BUDGET_RTOL * b[0], f
        s.close()
    assert failed > 3
