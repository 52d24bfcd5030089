"""Lloyd's sums over runs of equal labels (add_runs): a lane holds four consecutive points and a warp
128, so runs are cut inside lanes, at lanes, at warps and at the end of the points.  Coordinates
are multiples of 2^-10, so every binary64 sum is exact and the centres are the oracle's bits; the
clusters lie far apart, so no label is near a tie."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [7, 63, 127, 128, 129, 131, 1024, 1031, 5003])
@pytest.mark.parametrize("longest", [1, 3, 9, 300])
def test_runs_of_labels(n, longest):
    from paper_2307_00071_gb300 import gira
    rng = np.random.default_rng(n * 1000 + longest)
    k = 5
    runs = []
    while sum(map(len, runs)) < n:
        runs.append(np.full(rng.integers(1, longest + 1), rng.integers(k)))
    which = np.concatenate(runs)[:n]
    corners = 16.0 * np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1], [1, 1, 1]])
    pts = (corners[which] + rng.integers(-512, 513, size=(n, 3)) / 1024.0).astype(np.float32)
    c0, _ = oracle.kmeanspp(pts, k, 1)
    ref_c, ref_lab, ref_done = oracle.lloyd(pts, c0, 6)
    c, lab, done = gira.gira_kmeans_init(pts, k, seed=1, lloyd_iters=6)
    assert done == ref_done
    np.testing.assert_array_equal(np.asarray(lab), ref_lab)
    np.testing.assert_array_equal(np.asarray(c), ref_c.astype(np.float32))
