"""The E-step over reach lists (reach_kernels.cu) at the sizes where its tiling changes: blocks of
128 points, two or four warps per block (155,648 points), slices of 4,096 points in the statistics,
odd and padded component counts, and blocks holding a few or many points whose every component
lies more than 100 binades below the reference (listed again about the block's own maximum), also
points that no component's first list reaches.

Tolerances: per-point log-likelihoods within the derived bound of _parity.per_point_bound (which
covers the summation order); one EM iteration within the fit's 1e-4 per component.  The points
off the model there sit at q' of a few hundred, where the binary32 rounding of q' (a few 2^-24
relative) moves a responsibility by less than 1e-4.
"""
import numpy as np
import pytest

import oracle
from paper_2307_00071_gb300 import synth
from tests._parity import LL_ABS, assert_model_close, per_point_bound, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gira():
    from paper_2307_00071_gb300 import gira as g
    return g


@pytest.fixture(scope="module")
def frame():
    return synth.depth_frame(seed=4).points


def ball_model(pts, k, rng, d=3, sigma=0.05):
    """k isotropic components at scan points, with a jitter of their axes."""
    means = pts[rng.choice(len(pts), k, replace=False)].astype(np.float64)
    a = rng.normal(scale=0.2, size=(k, d, d))
    covs = sigma ** 2 * (np.eye(d) + a @ np.transpose(a, (0, 2, 1)))
    return rng.dirichlet(np.ones(k) * 5).astype(np.float32), means.astype(np.float32), covs.astype(np.float32)


def off_model(pts, count, rng):
    """count points of the cloud moved 0.8-1 m away, next to one another in the cloud's order."""
    at = rng.integers(0, len(pts) - count) + np.arange(count)
    out = pts.copy()
    step = rng.normal(size=(count, 3))
    out[at, :3] += (step / np.linalg.norm(step, axis=1)[:, None] * rng.uniform(0.8, 1.0, (count, 1))).astype(np.float32)
    return out, at


SIZES = [(1_100, 1_025, 0), (4_097, 1_500, 3), (38_912, 1_026, 16), (155_649, 1_099, 200), (12_289, 8_192, 700)]


@pytest.mark.parametrize("n,k,off", SIZES)
def test_large_k_reach(gira, frame, n, k, off):
    rng = np.random.default_rng(n + k)
    start = rng.integers(0, len(frame) - n)
    pts, at = off_model(np.ascontiguousarray(frame[start:start + n]), off, rng)
    w, m, c = ball_model(pts, k, rng)
    mean, pp = gira.gira_gmm_loglik(pts, w, m, c, per_point=True)
    pp = to_np(pp).astype(np.float64)
    assert mean == pytest.approx(pp.mean(), rel=1e-6)
    sample = np.unique(np.concatenate([at, [0, n - 1], rng.choice(n, 200, replace=False)]))
    _, _, lse = oracle.estep(pts[sample], w, m, c, want_resp=False, want_lse=True)
    err, bound = np.abs(pp[sample] - lse), per_point_bound(pts[sample], w, m, c)
    assert np.all(err <= bound), np.max(err / bound)
    r = gira.gira_gmm_fit(pts, k, iters=1, tol=0.0, init=(w, m, c))
    ref = oracle.em_par(pts, w, m, c, iters=1, tol=0.0, reg=1e-6)
    assert abs(r["trace"][0] - ref["trace"][0]) <= LL_ABS + 1e-7 * abs(ref["trace"][0])
    assert_model_close((r["weights"], r["means"], r["covs"]), (ref["weights"], ref["means"], ref["covs"]))


@pytest.mark.parametrize("n,k,off", [(1, 1, 0), (129, 3, 5), (5_000, 63, 300), (4_096, 64, 4_096), (20_001, 1_024, 900)])
def test_gradient_reach(gira, frame, n, k, off):
    """The gradients of a scan partly (or wholly) off the model against the oracle's: on one scan, and in a
    batch over reach lists (with and without the statistics launch)."""
    from tests.test_gpu_grad import assert_group, assert_points, check_all, ll_tol, pose12, ref_grads, rot
    rng = np.random.default_rng(n + k)
    start = rng.integers(0, len(frame) - n)
    pts = np.ascontiguousarray(frame[start:start + n])
    if off:
        pts, _ = off_model(pts, min(off, n - 1), rng)
    w, m, c = ball_model(frame[start:start + max(n, k)], k, rng)
    chol = np.linalg.cholesky(c.astype(np.float64)).astype(np.float32)
    R, t = rot(rng.normal(scale=0.02, size=3)).astype(np.float32), rng.normal(scale=0.02, size=3).astype(np.float32)
    args, ref = (pts, np.log(w), m, chol, pose12(R, t)), ref_grads(pts, np.log(w), m, chol, R, t)
    check_all(gira.gira_gmm_loglik_grad(*args), ref, n)
    twice = [np.concatenate([pts, pts]), [0, n, 2 * n], [k, k], *(np.concatenate([a, a]) for a in args[1:4]),
             np.stack([args[4], args[4]])]
    r = gira.gira_gmm_loglik_grad_batched(*twice, want=("points", "pose", "twist", "logits", "means"))
    only = gira.gira_gmm_loglik_grad_batched(*twice, want=("twist",))   # no statistics launch
    assert np.array_equal(to_np(only["grad_twist"]), to_np(r["grad_twist"])) and np.array_equal(only["loglik"], r["loglik"])
    for i in range(2):
        assert abs(r["loglik"][i] - ref["loglik"]) <= ll_tol(ref["loglik"], n)
        for g, per in (("logits", k), ("means", k), ("twist", 0), ("pose", 0)):
            got = to_np(r["grad_" + g])
            assert_group(got[i * k:(i + 1) * k] if per else got[i], ref["grad_" + g], g)
        assert_points(to_np(r["grad_points"])[i * n:(i + 1) * n], ref["grad_points"])


@pytest.mark.parametrize("n,k,off", [(1, 1, 0), (127, 2, 0), (4_097, 33, 5), (30_001, 1_023, 128), (8_193, 1_025, 600)])
def test_4d_reach(gira, frame, n, k, off):
    """Per-point log-likelihoods and one EM iteration in four dimensions."""
    rng = np.random.default_rng(n + k)
    start = rng.integers(0, len(frame) - n)
    full = np.concatenate([frame, synth.frame_intensity(frame)[:, None]], axis=1)
    pts = np.ascontiguousarray(full[start:start + n])
    at = np.zeros(0, np.int64)
    if off:
        pts, at = off_model(pts, off, rng)
    w, m, c = ball_model(full[start:start + max(n, k)], k, rng, d=4)
    mean, pp = gira.gira_gmm_loglik4(pts, w, m, c, per_point=True)
    pp = to_np(pp).astype(np.float64)
    sample = np.unique(np.concatenate([at, [0, n - 1], rng.integers(0, n, 200)]))
    _, _, lse = oracle.estep(pts[sample], w, m, c, want_resp=False, want_lse=True)
    err, bound = np.abs(pp[sample] - lse), per_point_bound(pts[sample], w, m, c, form="d")
    assert np.all(err <= bound), np.max(err / bound)
    r = gira.gira_gmm_fit4(pts, k, iters=1, tol=0.0, init=(w, m, c))
    ref = oracle.em(pts, w, m, c, iters=1, tol=0.0, reg=1e-6)
    assert abs(r["trace"][0] - ref["trace"][0]) <= LL_ABS + 1e-7 * abs(ref["trace"][0])
    assert_model_close((r["weights"], r["means"], r["covs"]), (ref["weights"], ref["means"], ref["covs"]))


@pytest.mark.parametrize("m,k", [(8191, 37), (8192, 1), (8193, 640), (8449, 2101)])
def test_regression_does_not_depend_on_the_order_of_the_locations(gira, frame, m, k):
    """The regression visits only the components that can have nonzero weight, listed for 256 and
    64 locations at a time (grouped by cell from 8,192 locations on, in rounds of 2,048 components).
    A location's result is that of its own components in increasing order, so it is the same bits
    in any order and in a call of a few locations; far locations make their neighbours' lists long.
    Against the oracle: locations at the surface (log-weights of size ~100, rounded to ~1e-5 of
    each weight), with the tolerances of the regression's own test."""
    rng = np.random.default_rng(m)
    pts4 = np.concatenate([frame, np.sin(3 * frame[:, :1])], 1).astype(np.float32)
    w, mu, cov = ball_model(pts4, k, rng, d=4, sigma=0.1)
    locs = frame[rng.choice(len(frame), m, replace=len(frame) < m)].astype(np.float32)
    far = rng.choice(m, 40, replace=False)
    locs[far] += rng.uniform(-30, 30, size=(40, 3)).astype(np.float32)
    e, v = (to_np(a) for a in gira.gira_gmm_conditional4(locs, w, mu, cov))
    p = rng.permutation(m)
    ep, vp = (to_np(a) for a in gira.gira_gmm_conditional4(locs[p], w, mu, cov))
    np.testing.assert_array_equal(ep, e[p])
    np.testing.assert_array_equal(vp, v[p])
    for a in (far[:7], np.arange(m - 300, m)):
        ea, va = (to_np(t) for t in gira.gira_gmm_conditional4(locs[a], w, mu, cov))
        np.testing.assert_array_equal(ea, e[a])
        np.testing.assert_array_equal(va, v[a])
    near = np.setdiff1d(np.arange(m), far)[:500]
    near = near[np.min(np.linalg.norm(locs[near, None] - mu[None, :, :3], axis=2), axis=1) < 0.5]
    re, rv = oracle.conditional4(locs[near], w, mu, cov)
    np.testing.assert_allclose(e[near], re, rtol=0, atol=2e-4)
    np.testing.assert_allclose(v[near], rv, rtol=2e-3, atol=2e-5)


@pytest.mark.parametrize("ks", [[416] * 24, [33, 1024, 129, 512, 1, 128] * 10])
def test_models_of_a_large_batch_equal_those_of_small_ones(gira, frame, ks):
    """From 305 blocks of 32 components on (here K_max / 32 per instance) a batch of gradients builds
    128 components per block: the same operations per component, so the same bits as in batches
    below that, also for odd K and in the last warps."""
    rng = np.random.default_rng(len(ks))
    ns = [1100 + 7 * i for i in range(len(ks))]
    assert (max(ks) + 31) // 32 * len(ks) > 304
    pts = [frame[rng.choice(len(frame), n, replace=False)] for n in ns]
    models = [ball_model(frame, k, rng) for k in ks]
    lg = [np.log(w) for w, _, _ in models]
    mu = [m for _, m, _ in models]
    ch = [np.linalg.cholesky(c.astype(np.float64)).astype(np.float32) for _, _, c in models]
    pose = np.tile(np.concatenate([np.eye(3).ravel(), [0.01, 0.0, 0.02]]).astype(np.float32), (len(ks), 1))

    def call(a, b):
        offs = np.concatenate([[0], np.cumsum(ns[a:b])]).astype(np.int64)
        return gira.gira_gmm_loglik_grad_batched(
            np.concatenate(pts[a:b]), offs, np.array(ks[a:b], np.int32), np.concatenate(lg[a:b]),
            np.concatenate(mu[a:b]), np.concatenate(ch[a:b]), pose[a:b], want=("twist", "means"))

    big = call(0, len(ks))
    at = np.concatenate([[0], np.cumsum(ks)])
    for a in range(0, len(ks), 6):
        part = call(a, a + 6)
        np.testing.assert_array_equal(np.asarray(part["loglik"]), np.asarray(big["loglik"])[a:a + 6])
        np.testing.assert_array_equal(to_np(part["grad_twist"]), to_np(big["grad_twist"])[a:a + 6])
        np.testing.assert_array_equal(to_np(part["grad_means"]), to_np(big["grad_means"])[at[a]:at[a + 6]])


@pytest.mark.parametrize("k,n", [(64, 3000), (65, 200_000), (64, 260_000), (256, 3000), (257, 3000)])
def test_batched_gradient_on_both_sides_of_the_dense_rule(gira, frame, k, n):
    """Batches of little dense work (at most 64 components and 500,000 points together, or 256 and
    16M pairs) take the dense kernel, others the reach lists; the same gradients as the single calls, which are dense: sums of n binary32
    terms in another order (a few 1e-6 of the sum of magnitudes, bounded by 2e-5 of the largest)."""
    rng = np.random.default_rng(k + n)
    pts = frame[rng.choice(len(frame), n, replace=False)]
    w, mu, cov = ball_model(frame, k, rng, sigma=0.2)
    lg, ch = np.log(w), np.linalg.cholesky(cov.astype(np.float64)).astype(np.float32)
    want = ("twist", "means", "points")
    one = gira.gira_gmm_loglik_grad(pts, lg, mu, ch, None, want=want)
    two = gira.gira_gmm_loglik_grad_batched(np.concatenate([pts, pts]), np.array([0, n, 2 * n], np.int64),
                                            np.array([k, k], np.int32), np.concatenate([lg, lg]),
                                            np.concatenate([mu, mu]), np.concatenate([ch, ch]), want=want)
    assert two["loglik"][1] == pytest.approx(one["loglik"], rel=1e-6)
    for key, rows in (("grad_twist", 1), ("grad_means", k), ("grad_points", n)):
        a = to_np(one[key]).astype(np.float64)
        b = to_np(two[key]).astype(np.float64).reshape(2, *a.shape)[1]
        assert np.max(np.abs(a - b)) <= 2e-5 * np.max(np.abs(a)), key


@pytest.mark.parametrize("d", [3, 4])
@pytest.mark.parametrize("n,k,off", [(1_025, 1_025, 0), (8_193, 8_192, 40), (38_912, 1_101, 300), (38_913, 1_101, 300),
                                     (2_000, 511, 7), (2_000, 512, 7), (2_000, 1_537, 1_999)])
def test_shuffled_scores(gira, frame, d, n, k, off):
    """The log-likelihood of points in no order, where a block's box is the whole scene: sixteen warps share
    a block up to 304 blocks (from 512 components), four above.  Points off the model take the exact maximum."""
    rng = np.random.default_rng(n + k)
    full = np.concatenate([frame, synth.frame_intensity(frame)[:, None]], axis=1)[:, :d]
    pts, at = off_model(np.ascontiguousarray(full[rng.integers(0, len(full) - n) + np.arange(n)]), off, rng) if off else (
        np.ascontiguousarray(full[:n]), np.zeros(0, np.int64))
    w, m, c = ball_model(full, k, rng, d=d)
    order = rng.permutation(n)
    call = gira.gira_gmm_loglik if d == 3 else gira.gira_gmm_loglik4
    mean, pp = call(np.ascontiguousarray(pts[order]), w, m, c, per_point=True)
    back = np.empty(n)
    back[order] = to_np(pp)
    assert mean == pytest.approx(back.mean(), rel=1e-6)
    sample = np.unique(np.concatenate([at[:100], [0, n - 1], rng.choice(n, min(n, 200), replace=False)]))
    _, _, lse = oracle.estep(pts[sample], w, m, c, want_resp=False, want_lse=True)
    err, bound = np.abs(back[sample] - lse), per_point_bound(pts[sample], w, m, c, form="d" if d == 4 else "b")
    assert np.all(err <= bound), np.max(err / bound)


@pytest.mark.parametrize("ns,ks", [([5_000], [512]), ([5_000], [1_024]), ([300], [300]), ([2_500] * 4, [1_024] * 4),
                                   ([2_500] * 5, [1_024] * 5), ([30_001, 2_000], [300, 1_023]),
                                   ([5_000] * 9 + [1_500], [32] * 9 + [1_024])])
def test_batched_gradient_of_few_scans_with_large_models(gira, frame, ns, ks):
    """Above 256 components a few small scans, and batches with hardly a point under a large model, take the
    dense kernel, others the reach lists: the same gradients as the single calls, within the rounding of
    sums of n binary32 terms in another order (2e-5 of the largest)."""
    rng = np.random.default_rng(sum(ns) + sum(ks))
    pts = [frame[rng.choice(len(frame), n, replace=False)] for n in ns]
    models = [ball_model(frame, k, rng, sigma=0.2) for k in ks]
    lg, mu = [np.log(w) for w, _, _ in models], [m for _, m, _ in models]
    ch = [np.linalg.cholesky(c.astype(np.float64)).astype(np.float32) for _, _, c in models]
    want = ("twist", "logits", "means", "points")
    r = gira.gira_gmm_loglik_grad_batched(np.concatenate(pts), np.concatenate([[0], np.cumsum(ns)]).astype(np.int64),
                                          np.array(ks, np.int32), np.concatenate(lg), np.concatenate(mu),
                                          np.concatenate(ch), want=want)
    at = {"grad_points": np.concatenate([[0], np.cumsum(ns)]), "grad_twist": np.arange(len(ns) + 1)}
    comps = np.concatenate([[0], np.cumsum(ks)])
    for i, n in enumerate(ns):
        one = gira.gira_gmm_loglik_grad(pts[i], lg[i], mu[i], ch[i], None, want=want)
        assert r["loglik"][i] == pytest.approx(one["loglik"], rel=1e-6)
        for key in ("grad_twist", "grad_logits", "grad_means", "grad_points"):
            a = to_np(one[key]).astype(np.float64)
            b = to_np(r[key]).astype(np.float64)
            lo, hi = at.get(key, comps)[i:i + 2]
            b = b.reshape(-1, 6)[i] if key == "grad_twist" else b[lo:hi]
            assert np.max(np.abs(a - b.reshape(a.shape))) <= 2e-5 * np.max(np.abs(a)), key
