"""Directions of merged rays that have split to levels beyond the pixel table:
every child's direction is its pixel's centre on its merge cell's sphere."""
import dataclasses as dc

import numpy as np
import pytest

import oracle
import paper_2409_04521_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu


def test_children_of_merged_rays_beyond_the_pixel_table():
    # the batch's table ends at level 6 (its own N_min); the member's larger
    # N_min splits its rays, merged ones among them, to deeper levels
    p = W.batch_member(3, sizes=(16,), nsteps=14)
    p = dc.replace(p, options=dc.replace(p.options, n_ray_min=200.0, merge=True, n_ex=0.5, l_merge=1))
    b = F.Batch(max_sims=2, max_grid=16, nbins=3, ray_capacity=1 << 22, cell_capacity=2 * 16 ** 3,
                emitter_capacity=128, n_ray_min=3.0, merge_l_max=1)
    slot = b.add(p)
    seen = 0
    o = p.options
    for k in range(p.nsteps):
        b.step()
        r = b.rays(slot)
        deep = np.nonzero(r["merged"] & ~r["vertex"] & (r["level"] > 6))[0]
        seen += len(deep)
        for i in deep[:: max(1, len(deep) // 200)]:
            Rq = oracle.merge_rotation(o.seed, int(r["emitter"][i]) - (1 << 31), int(r["birth"][i]), o.rotate)
            assert np.array_equal(r["dir"][i], oracle.direction(int(r["level"][i]), int(r["pixel"][i]), Rq)), (k, i)
    assert seen > 0
    b.close()
