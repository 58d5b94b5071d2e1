"""The march's record tiles over many rounds of a warp: a warp's tile is
rewritten by its splitting lanes and refilled by the next copy, so few warps
must march and split the same rays as many."""
import dataclasses as dc

import numpy as np
import pytest

import paper_2409_04521_gb300 as F
import workloads as W
from parity_util import RAY_RTOL, ray_table

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("nb", [1, 4, 7])
def test_few_warps_march_and_split_the_rays_of_many(nb):
    p = W.cosmo16(n=40, nsteps=20, nsrc=16, seed=9)
    sp = W.blackbody_bins(1e5, 13.6 * 4.0 ** (np.arange(nb + 1) / nb))
    # (no terminations: those within rounding of the threshold may differ)
    p = dc.replace(p, spectrum=sp, options=dc.replace(p.options, eps_term=0.0))
    many, few = F.Simulation(p, ray_capacity=1 << 21), F.Simulation(p, ray_capacity=1 << 21)
    few.set_launch(0, 2, 1, 128)                       # four warps an SM
    for _ in range(p.nsteps):
        many.step(p.dt)
        few.step(p.dt)
    (ka, da, na), (kb, db, nb_) = ray_table(many.rays()), ray_table(few.rays())
    assert len(ka) > 4 * 32 * 4 * 152                  # more than four rounds a warp
    assert np.array_equal(ka, kb) and np.array_equal(da, db)
    # two runs differ by the order of their deposits only (RAY_RTOL holds for
    # a run against the oracle; far weaker rays have more opacity behind them)
    big = na > 1e-9 * na.max()
    assert np.all(np.abs(na - nb_)[big] <= RAY_RTOL * na[big])
    many.close()
    few.close()
