"""Deposits of two words a cell (one simulation, isothermal, without segment
counts) against the oracle, and beside the four-word deposits of the same run
with segment counts; the tolerances are those of the other parity runs."""
import dataclasses as dc

import numpy as np
import pytest

import oracle
import paper_2409_04521_gb300 as F
import workloads as W
from parity_util import budget_checks, compare_fields

pytestmark = pytest.mark.gpu


def _iso(p, **kw):
    return dc.replace(p, options=dc.replace(p.options, isothermal=True, T_init=1e4, **kw))


@pytest.mark.parametrize("prob", [W.stromgren(n=16, nsteps=12), W.cosmo20k(n=24, nsteps=8, nsrc=40),
                                  _iso(W.cosmo16(n=20, nsteps=8, nsrc=5)),
                                  _iso(W.cosmo16(n=16, nsteps=6, nsrc=3), gamma_iters=3)],
                         ids=["one bin", "three bins, mfp law", "four bins", "three passes"])
def test_two_word_deposits(prob):
    g = F.Simulation(prob, ray_capacity=1 << 20)
    d = F.Simulation(prob, ray_capacity=1 << 20, keep_diagnostics=True)
    o = oracle.OracleSim(prob)
    for k in range(prob.nsteps):
        if k == 3:
            g.set_launch(1, 2)                     # an aggregating variant deposits four words
        if k == 4:
            g.set_launch(0, 3)
        for s in (g, d, o):
            s.step(prob.dt)
    assert g.counts()["segments_total"] == d.counts()["segments_total"]
    for s in (g, d):
        compare_fields(s.fields(), o.fields())
        budget_checks(s.budget(), o.budget())
    assert np.array_equal(g.fields(("T",))["T"], d.fields(("T",))["T"])
    for s in (g, d, o):
        s.close()
