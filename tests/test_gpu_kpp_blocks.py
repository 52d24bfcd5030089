"""k-means++ over sub-blocks in L2 (kpp_blocks_kernel): the drawn centres are the oracle's bit for
bit, at one point per warp and less, ragged last sub-blocks, several sub-blocks per warp and per
lane of the search, weights above 2^10 (128-bit totals), all-zero weights, and a shuffled cloud of
the same size, which takes another kernel."""
import numpy as np
import pytest

import oracle
from paper_2307_00071_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gira():
    from paper_2307_00071_gb300 import gira as g
    return g


@pytest.fixture(scope="module")
def frames():
    return np.concatenate([synth.depth_frame(seed=s).points for s in (5, 6)])


def seeds(gira, pts, k, seed):
    """The seeding alone (no Lloyd update): 3-D centres, or a 4-D fit's one-hot means of it."""
    return np.asarray(gira.gira_kmeans_init(pts, k, seed=seed, lloyd_iters=0, want_labels=False)[0])


@pytest.mark.parametrize("n,k,scale,order", [(294_913, 40, 1.0, "sensor"), (500_001, 24, 1.0, "sensor"),
                                             (540_000, 12, 60.0, "sensor"), (300_000, 12, 1.0, "shuffled"),
                                             (300_001, 6, 0.0, "sensor")])
def test_large_3d(gira, frames, n, k, scale, order):
    pts = np.ascontiguousarray(frames[:n] * np.float32(scale))
    if order == "shuffled":
        pts = pts[np.random.default_rng(n).permutation(n)]
    assert np.array_equal(seeds(gira, pts, k, 3), oracle.kmeanspp(pts, k, 3)[0].astype(np.float32))


@pytest.mark.parametrize("n,k,scale", [(5, 5, 1.0), (33, 7, 1.0), (8_191, 30, 1.0), (70_001, 16, 1.0), (276_000, 16, 60.0),
                                       (9_000, 4, 0.0)])
def test_4d(gira, frames, n, k, scale):
    """KInit with Lloyd in four dimensions, no EM iteration: the one-hot model of the oracle's labels."""
    full = np.concatenate([frames[:n], synth.frame_intensity(frames[:n])[:, None]], axis=1) * np.float32(scale)
    full = np.ascontiguousarray(full.astype(np.float32))
    r = gira.gira_gmm_fit4(full, k, iters=0, seed=2, lloyd_iters=1, reg_covar=1e-3, final_loglik=False)
    ref = oracle.kinit(full, k, 2, 1, 1e-3)
    for key in ("weights", "means", "covs"):
        got, want = np.asarray(r[key], np.float64), np.asarray(ref[key], np.float64)
        assert np.all(np.abs(got - want) <= 2e-7 * np.abs(want).max() + 1e-12), key   # binary32 outputs


@pytest.mark.parametrize("n,k,lloyd", [(1, 1, 2), (130, 100, 3), (60_000, 700, 4), (20_000, 2_049, 2)])
def test_lloyd_4d(gira, frames, n, k, lloyd):
    """Pruned and full (above 2,048 centres) assignments: every label as the oracle's, so the one-hot weights
    (counts / n, exact to binary32) agree, and the model with them."""
    full = np.concatenate([frames[:n], synth.frame_intensity(frames[:n])[:, None]], axis=1).astype(np.float32)
    full = np.ascontiguousarray(full)
    r = gira.gira_gmm_fit4(full, k, iters=0, seed=4, lloyd_iters=lloyd, reg_covar=1e-3, final_loglik=False)
    ref = oracle.kinit(full, k, 4, lloyd, 1e-3)
    assert np.array_equal(np.rint(np.asarray(r["weights"], np.float64) * n), np.bincount(ref["labels"], minlength=k))
    for key in ("means", "covs"):
        got, want = np.asarray(r[key], np.float64), np.asarray(ref[key], np.float64)
        assert np.all(np.abs(got - want) <= 2e-7 * np.abs(want).max() + 1e-12), key


@pytest.mark.parametrize("dim,n,far", [(3, 300_001, [(7, 3e38)]), (3, 294_913, [(294_912, -1e20), (40, 1e20)]),
                                       (4, 5_000, [(4_999, 2e19)]), (4, 70_001, [(33, 1e20), (69_000, -1e20), (1, 3e38)])])
def test_overflowing_distances(gira, frames, dim, n, far):
    """Points so far away that D^2 is +inf (weight 2^95 - 1): drawn first, whatever an earlier call left in
    the workspace.  Bits in 3-D; in 4-D the counts, with every far point alone in its cluster."""
    pts = frames[:n] if dim == 3 else np.concatenate([frames[:n], synth.frame_intensity(frames[:n])[:, None]], axis=1)
    pts = pts.astype(np.float32)   # a copy
    k = 6
    other = np.repeat((np.arange(n, dtype=np.float32) % 977)[:, None], 4, axis=1)
    gira.gira_gmm_fit4(other, 4, iters=0, reg_covar=1e-3, final_loglik=False)   # other D^2 in the workspace
    for at, value in far:
        pts[at, at % dim] = value
    if dim == 3:
        assert np.array_equal(seeds(gira, pts, k, 5), oracle.kmeanspp(pts, k, 5)[0].astype(np.float32))
        return
    r = gira.gira_gmm_fit4(pts, k, iters=0, seed=5, lloyd_iters=0, reg_covar=1e-3, final_loglik=False)
    ref = oracle.kinit(pts, k, 5, 0, 1e-3)
    want = np.bincount(ref["labels"], minlength=k)
    assert sum(want == 1) >= len(far)
    assert np.array_equal(np.rint(np.asarray(r["weights"], np.float64) * n), want)
