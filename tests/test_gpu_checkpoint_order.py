"""A checkpoint of many rays: the load's copies reach the device before the
kernel that takes the ray arrays apart, however long they take."""
import numpy as np
import pytest

import paper_2409_04521_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu


def test_large_checkpoint_round_trip():
    p = W.cosmo16(n=64, nsteps=40, nsrc=16, seed=9)
    s = F.Simulation(p, ray_capacity=1 << 24)
    for _ in range(p.nsteps):
        s.step(p.dt)
    blob = s.save_state()
    assert s.counts()["rays"] * 40 > 16 << 20             # ten words a ray: more than any staging buffer
    t = F.Simulation(p, ray_capacity=1 << 24)
    for k in range(4):
        # a fresh pageable copy each time, into a state that has moved on
        t.load_state(blob.copy())
        assert np.array_equal(t.save_state(), blob), k
        t.step(p.dt)
    s.close()
    t.close()
