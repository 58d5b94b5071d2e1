"""Batches whose march needs more shared memory than a block gets unasked:
every slot count around that line, and batches of different sizes alive at
once."""
import dataclasses as dc

import numpy as np
import pytest

import paper_2409_04521_gb300 as F
import workloads as W

pytestmark = pytest.mark.gpu


def _prob(nbins, **kw):
    p = W.batch_member(2, sizes=(16,), nsteps=5)
    sp = W.blackbody_bins(1e5, 13.6 * 4.0 ** (np.arange(nbins + 1) / nbins))
    return dc.replace(p, spectrum=sp, options=dc.replace(p.options, **kw))


def _batch(slots, nbins, **kw):
    return F.Batch(max_sims=slots, max_grid=16, nbins=nbins, ray_capacity=1 << 18, cell_capacity=2 * 16 ** 3,
                   emitter_capacity=128, **kw)


def _run(b, p):
    s = b.add(p)
    for _ in range(p.nsteps):
        b.step()
    b.sync()
    return b.counts(s), b.fields(s)


def _alone(p):
    s = F.Simulation(p, ray_capacity=1 << 18)
    for _ in range(p.nsteps):
        s.step(p.dt)
    out = s.counts(), s.fields()
    s.close()
    return out


def _check(got, ref):
    (c, f), (rc, rf) = got, ref
    assert c["rays"] == rc["rays"] > 0 and c["segments_total"] == rc["segments_total"]
    # two runs differ by the order of their deposits: a few 1e-7 a step
    assert np.allclose(f["gamma_HI"], rf["gamma_HI"], rtol=1e-5, atol=1e-5 * rf["gamma_HI"].max())


# dynamic shared memory just below, on and just above 48 KB less the march's
# static part, and at the largest batch
@pytest.mark.parametrize("nbins,slots", [(1, 83), (1, 84), (1, 86), (3, 68), (3, 69), (3, 70), (4, 61), (4, 62),
                                         (8, 30), (8, 31), (8, 512)])
def test_every_slot_count_around_the_shared_memory_line(nbins, slots):
    p = _prob(nbins)
    b = _batch(slots, nbins)
    got = _run(b, p)
    b.close()
    _check(got, _alone(p))


@pytest.mark.parametrize("nbins,slots", [(3, 30), (4, 22), (6, 7)])
def test_the_same_in_merging_batches(nbins, slots):
    p = _prob(nbins)
    b = _batch(slots, nbins, merge_l_max=0)
    got = _run(b, p)
    b.close()
    _check(got, _alone(p))


@pytest.mark.parametrize("use_graph", [False, True])
def test_a_smaller_batch_leaves_a_larger_one_its_shared_memory(use_graph):
    p = _prob(4)
    big = _batch(128, 4, use_graph=use_graph)
    small = _batch(64, 4, use_graph=use_graph)
    ref = _alone(p)
    _check(_run(big, p), ref)
    _check(_run(small, p), ref)
    big.close()
    small.close()
