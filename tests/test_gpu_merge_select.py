"""The merge's radix select (Sec. 3.3): the K-th largest content, and with it
the exempt rays, for every K over contents that lie at the edges of the
select's segments (256 upper halves) and bins, some of them equal."""
import numpy as np
import pytest

import paper_2409_04521_gb300 as F

pytestmark = pytest.mark.gpu

HIGH = [0x3eff, 0x3f00, 0x3f01, 0x3fff, 0x4000]
LOW = [0x0000, 0x0001, 0x00ff, 0x0100, 0x7fff, 0xff00, 0xffff]


def test_exempt_rays_at_the_edges_of_segments_and_bins():
    bits = np.array([(h << 16) | l for h in HIGH for l in LOW] * 2, np.uint32)
    T = np.random.default_rng(3).permutation(bits).view(np.float32)
    n = len(T)
    # one cell and one direction: what is not exempt becomes one ray
    rays = dict(level=np.zeros(n), pixel=np.zeros(n), emitter=np.zeros(n), birth=np.zeros(n),
                dir=np.tile([1 << 19, 1 << 18, 1 << 20], (n, 1)), N=T[:, None])
    order = np.sort(T)[::-1]
    for K in range(1, n):
        ex = T[T >= order[K - 1]]
        rest = T[T < order[K - 1]]
        if len(rest) == 1:
            ex, rest = T, T[:0]                        # a ray alone in its group stays
        out = F.probe_merge((4, 4, 4), 1, 0, 12, 0, K, 7, 1, 0, 1e-10, [[1, 1, 1]], [1.0], rays)
        m = out["merged"]
        assert np.array_equal(np.sort(out["N"][~m, 0]), np.sort(ex).astype(np.float64)), K
        assert m.sum() == (1 if len(rest) else 0), K
        if len(rest):
            # a single-precision sum of at most 70 contents
            assert np.isclose(out["N"][m, 0], rest.astype(np.float64).sum(), rtol=70 * 2.0 ** -24), K
