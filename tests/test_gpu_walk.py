"""One-step traversal where two face crossings lie so close that the walk's
single-precision times cannot order them: the crossed cells stay those of the
exact segment, and the lengths within five single-precision ulp (two
approximate reciprocals, three products and the difference's 1.5 ulp)."""
import numpy as np
import pytest

import oracle
import paper_2409_04521_gb300 as F

S = 2 ** 21


def _rays(gap, seed):
    """Rays whose x, y (and for a third of them z) crossings are about `gap`
    (in units of the step) apart, some of them at the very end of the step."""
    rng = np.random.default_rng(seed)
    p0, d = [], []
    for i in range(600):
        a = rng.integers(S // 64, S, 3)
        if i % 5 == 0:
            a[1] = a[0]                                    # exact ties are possible
        t = rng.uniform(0.0, 0.95) if i % 3 else 1.0 - 2.0 / S
        D = np.empty(3, np.int64)
        D[0] = max(1, min(a[0] - 1, int(t * a[0])))
        for k in (1, 2):
            D[k] = np.rint((D[0] / a[0] + rng.choice([-1, 1]) * gap) * a[k]) + rng.integers(-1, 2)
        if i % 3 == 1:
            D[2] = rng.integers(1, S + 1)
        D = np.clip(D, 1, S)
        sg = rng.choice([-1, 1], 3)
        c = rng.integers(0, 4, 3)
        p0.append(np.where(sg > 0, (c + 1) * S - D, c * S + D))
        d.append(sg * a)
    return np.array(p0, np.int64), np.array(d, np.int64)


@pytest.mark.gpu
@pytest.mark.parametrize("gap", [0.0, 2.0 ** -23, 2.0 ** -21, 2.0 ** -20, 2.0 ** -19, 2.0 ** -16])
def test_close_crossings_keep_the_exact_cells(gap):
    grid = (4, 3, 5)
    p0, d = _rays(gap, 17)
    cells, ds, nseg, esc = F.probe_traverse(p0, d, grid)
    for i in range(len(p0)):
        oc, ods, oesc = oracle.traverse(p0[i], d[i], grid)
        k = len(oc)
        assert nseg[i] == k and bool(esc[i]) == oesc, i
        assert np.array_equal(cells[i, :k], oc), i
        assert np.allclose(ds[i, :k], ods, rtol=6e-7, atol=0), (i, ds[i, :k], ods)
