"""Lloyd's sums over runs of equal labels (add_runs): a lane holds four consecutive points and a warp
128, so runs are cut inside lanes, at lanes, at warps and at the end of the points.  Coordinates
are multiples of 2^-10, so every binary64 sum is exact and the centres are the oracle's bits; the
clusters lie far apart, so no label is near a tie."""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu


def runs_of_points(n, longest):
    rng = np.random.default_rng(n * 1000 + longest)
    runs = []
    while sum(map(len, runs)) < n:
        runs.append(np.full(rng.integers(1, longest + 1), rng.integers(5)))
    which = np.concatenate(runs)[:n]
    corners = 16.0 * np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1], [1, 1, 1]])
    return (corners[which] + rng.integers(-512, 513, size=(n, 3)) / 1024.0).astype(np.float32)


@pytest.mark.parametrize("n", [7, 63, 127, 128, 129, 131, 1024, 1031, 5003])
@pytest.mark.parametrize("longest", [1, 3, 9, 300])
def test_runs_of_labels(n, longest):
    from paper_2307_00071_gb300 import gira
    k = 5
    pts = runs_of_points(n, longest)
    c0, _ = oracle.kmeanspp(pts, k, 1)
    ref_c, ref_lab, ref_done = oracle.lloyd(pts, c0, 6)
    c, lab, done = gira.gira_kmeans_init(pts, k, seed=1, lloyd_iters=6)
    assert done == ref_done
    np.testing.assert_array_equal(np.asarray(lab), ref_lab)
    np.testing.assert_array_equal(np.asarray(c), ref_c.astype(np.float32))


@pytest.mark.parametrize("n", [255, 256, 513, 2051, 70001])
@pytest.mark.parametrize("batched", [False, True])
def test_one_hot_statistics_of_runs(n, batched):
    """The statistics that start EM, summed over runs the same way (eight points per lane; small
    blocks up to 65,536 points): the model of a fit without iterations.  Binary64 throughout, so
    within two roundings of the binary32 outputs."""
    from paper_2307_00071_gb300 import gira
    pts = [runs_of_points(n, 9)] + ([runs_of_points(301, 3)] if batched else [])
    for p in pts:
        assert len(np.unique(np.round(p / 16.0), axis=0)) == 5
    opts = dict(iters=0, tol=0.0, reg_covar=1e-3, seed=1, lloyd_iters=2)
    if batched:
        offs = np.cumsum([0] + [len(p) for p in pts]).astype(np.int64)
        r = gira.gira_gmm_fit_batched(np.concatenate(pts), offs, np.array([5, 5], np.int32), **opts)
    else:
        r = gira.gira_gmm_fit(pts[0], 5, **opts)
    for i, p in enumerate(pts):
        ref = oracle.kinit(p, 5, 1, 2, 1e-3)
        for key in ("weights", "means", "covs"):
            got = np.asarray(r[key], np.float64)[5 * i:5 * i + 5]
            np.testing.assert_allclose(got, ref[key], rtol=1.2e-7, atol=1e-8)


@pytest.mark.parametrize("clusters", [2, 3, 4, 5])
@pytest.mark.parametrize("n", [130, 1031, 40_007])
def test_labels_in_no_order(n, clusters):
    """Dozens of runs a warp: up to four labels are summed over the warp, more by runs; exact sums, so the
    oracle's bits, in three and (the one-hot model) four dimensions."""
    from paper_2307_00071_gb300 import gira
    rng = np.random.default_rng(n + clusters)
    corners = 16.0 * np.array([[0, 0, 0], [1, 0, 0], [0, 1, 0], [0, 0, 1], [1, 1, 1]])[:clusters]
    pts = (corners[rng.integers(clusters, size=n)] + rng.integers(-512, 513, size=(n, 3)) / 1024.0).astype(np.float32)
    c0, _ = oracle.kmeanspp(pts, clusters, 1)
    ref_c, ref_lab, ref_done = oracle.lloyd(pts, c0, 6)
    c, lab, done = gira.gira_kmeans_init(pts, clusters, seed=1, lloyd_iters=6)
    assert done == ref_done
    np.testing.assert_array_equal(np.asarray(lab), ref_lab)
    np.testing.assert_array_equal(np.asarray(c), ref_c.astype(np.float32))
    full = np.concatenate([pts, rng.integers(0, 1025, size=(n, 1)) / 1024.0], axis=1).astype(np.float32)
    r = gira.gira_gmm_fit4(full, clusters, iters=0, seed=1, lloyd_iters=3, reg_covar=1e-3, final_loglik=False)
    ref = oracle.kinit(full, clusters, 1, 3, 1e-3)
    for key in ("weights", "means", "covs"):
        np.testing.assert_allclose(np.asarray(r[key], np.float64), ref[key], rtol=1.2e-7, atol=1e-7)


def test_near_ties():
    """Points around the plane half way between two centres: a label is the nearer centre, or one whose
    distance agrees with it to 2^-21 (D^2 in binary32: four roundings, fused or not, on both sides)."""
    from paper_2307_00071_gb300 import gira
    rng = np.random.default_rng(7)
    m = 50_000
    a, b = rng.uniform(-1, 1, size=(2, 3)).astype(np.float32)
    u = b.astype(np.float64) - a
    u /= np.linalg.norm(u)
    t = rng.normal(size=(m, 3))
    t -= (t @ u)[:, None] * u
    probes = (a.astype(np.float64) + b) / 2 + t + rng.normal(scale=1e-7, size=(m, 1)) * u
    pts = np.concatenate([np.tile(a, (m, 1)), np.tile(b, (m, 1)), probes]).astype(np.float32)
    c, lab, _ = gira.gira_kmeans_init(pts, 2, seed=0, lloyd_iters=0)
    d = ((pts.astype(np.float64)[:, None] - np.asarray(c, np.float64)[None]) ** 2).sum(2)
    mine = np.take_along_axis(d, np.asarray(lab, np.int64)[:, None], 1)[:, 0]
    assert np.all(mine <= d.min(1) * (1 + 2.0 ** -21))
