"""The ray queue's record layout at every bin count, and emission around the
edges of a warp of emitters, against the oracle; the checkpoint's ray arrays
keep one array a word."""
import dataclasses as dc
import os
import subprocess
import sys

import numpy as np
import pytest

import paper_2409_04521_gb300 as F
import workloads as W
from parity_util import ray_table, run_pair

pytestmark = pytest.mark.gpu


def _prob(nb, nsrc, l_src=0, n=14, nsteps=5):
    p = W.cosmo16(n=n, nsteps=nsteps, nsrc=nsrc, seed=5)
    sp = W.blackbody_bins(1e5, 13.6 * 4.0 ** (np.arange(nb + 1) / nb))
    return dc.replace(p, spectrum=sp, options=dc.replace(p.options, l_src=l_src, n_ray_min=2.0))


# tolerances: those of the other parity runs (T as the temperature runs there)
@pytest.mark.parametrize("nb", range(1, 9))
@pytest.mark.parametrize("nsrc,l_src", [(1, 0), (33, 1)])
def test_records_and_emission(nb, nsrc, l_src):
    run_pair(_prob(nb, nsrc, l_src), T_rtol=2e-3)


@pytest.mark.parametrize("nsrc", [31, 32, 70])
def test_emission_at_the_edges_of_a_warp(nsrc):
    run_pair(_prob(4, nsrc), T_rtol=2e-3)


@pytest.mark.parametrize("nb", [1, 3, 6, 8])
def test_checkpoint_keeps_one_array_a_word(nb):
    p = _prob(nb, 3)
    s = F.Simulation(p, ray_capacity=1 << 18)
    for _ in range(4):
        s.step(p.dt)
    r = s.rays()
    n = len(r["level"])
    blob = s.save_state()
    w = blob[len(blob) - (6 + nb) * 4 * n:].view(np.uint32).reshape(6 + nb, n)
    assert np.array_equal(w[0], (r["level"].astype(np.uint32) << 28) | r["pixel"].astype(np.uint32))
    assert np.array_equal(w[1], r["emitter"].astype(np.uint32))
    assert np.array_equal(w[2], r["birth"].astype(np.uint32))
    assert np.array_equal(w[3:6].view(np.int32), r["dir"].T)
    ph = w[6:].view(np.float32).astype(np.float64)
    k = r["N"].T / np.where(ph > 0, ph, 1.0)              # one power of two: photons per code photon
    assert np.all((ph > 0) == (r["N"].T > 0)) and np.unique(k[ph > 0]).size == 1
    t = F.Simulation(p, ray_capacity=1 << 18)
    t.load_state(blob)
    assert np.array_equal(t.save_state(), blob)
    s.close()
    t.close()


def test_children_beyond_the_batch_pixel_table():
    # the batch's table is sized by its own N_min; a member with a larger one
    # splits deeper, past the table, and must get the directions it gets alone
    p = W.batch_member(3, sizes=(16,), nsteps=9)
    p = dc.replace(p, options=dc.replace(p.options, n_ray_min=200.0))
    b = F.Batch(max_sims=2, max_grid=16, nbins=3, ray_capacity=1 << 22, cell_capacity=2 * 16 ** 3,
                emitter_capacity=128, n_ray_min=3.0)
    slot = b.add(p)
    s = F.Simulation(p, ray_capacity=1 << 22)
    for _ in range(p.nsteps):
        b.step()
        s.step(p.dt)
    kb, db, _ = ray_table(b.rays(slot))
    ks, ds, _ = ray_table(s.rays())
    assert ks[:, 2].max() >= 7                            # table levels 0..6
    assert np.array_equal(kb, ks) and np.array_equal(db, ds)
    b.close()
    s.close()


_TWO_TABLES = """
import dataclasses as dc, sys
import numpy as np
sys.path[:0] = [%r, %r]
import paper_2409_04521_gb300 as F, workloads as W
from parity_util import ray_table
p = W.cosmo16(n=16, nsteps=8, nsrc=3, seed=5)
a = F.Simulation(p, ray_capacity=1 << 18)
a.step(p.dt)
a.sync()
# a simulation that splits deeper makes a deeper table; the first keeps its own
b = F.Simulation(dc.replace(p, options=dc.replace(p.options, n_ray_min=5000.0)), ray_capacity=1 << 18)
for _ in range(7):
    a.step(p.dt)
ka, da, _ = ray_table(a.rays())
c = F.Simulation(p, ray_capacity=1 << 18)
for _ in range(8):
    c.step(p.dt)
kc, dd, _ = ray_table(c.rays())
assert np.array_equal(ka, kc) and np.array_equal(da, dd)
print("same rays", len(ka))
"""


def test_a_deeper_pixel_table_leaves_the_older_one_to_its_simulation():
    # in a process of its own: the tables are the process's
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, "-c", _TWO_TABLES % (root, os.path.join(root, "tests"))], cwd=root,
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "same rays" in r.stdout, r.stdout + r.stderr
