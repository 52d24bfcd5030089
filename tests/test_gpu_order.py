"""The spatial order the fits' E-steps visit points in (a stable radix sort by
Morton code), through the test hook gira_test_point_order.

The expected order is computed here from the hook's documented rule: per
instance, the bounding box of its points, cells of (largest extent) / 64 on
every axis, cell index floor((x - lo) * (64 / extent)) clamped to [0, 63] in
binary32, the three 6-bit indices interleaved (bit 3b + a = bit b of axis a),
and a stable sort by (instance, code).  The E-step's results do not depend on
the order beyond the rounding of its sums; this pins the order itself.
"""
import numpy as np
import pytest

from paper_2307_00071_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def codes(pts):
    x = np.asarray(pts, np.float32)
    lo, hi = x.min(0), x.max(0)
    ext = np.float32(max(hi - lo))
    scale = np.float32(64.0) / ext if ext > 0 else np.float32(0.0)
    q = np.clip(np.floor((x - lo[None]).astype(np.float32) * scale), 0, 63).astype(np.int64)
    code = np.zeros(len(x), np.int64)
    for b in range(6):
        for a in range(3):
            code |= ((q[:, a] >> b) & 1) << (3 * b + a)
    return code


def expected(pts, offsets):
    out = []
    for i in range(len(offsets) - 1):
        a, b = offsets[i], offsets[i + 1]
        out.append(a + np.argsort(codes(pts[a:b]), kind="stable"))
    return np.concatenate(out)


def run(pts, offsets=None):
    from paper_2307_00071_gb300 import gira
    x = torch.as_tensor(np.ascontiguousarray(pts, np.float32), device="cuda")
    got = gira.gira_test_point_order(x, offsets).cpu().numpy()
    want = expected(np.asarray(pts, np.float32), [0, len(pts)] if offsets is None else list(offsets))
    np.testing.assert_array_equal(got, want)


def test_frame_order():
    run(synth.depth_frame(seed=1).points)


@pytest.mark.parametrize("n", [1, 31, 2049, 100_003])
def test_uniform_clouds_ragged_sizes(n):
    run(synth.uniform_cloud(n, seed=n, scale=3.0))


def test_repeated_and_degenerate_points():
    pts = np.zeros((5000, 3), np.float32)   # one point repeated: zero extent, every code 0
    run(pts)
    rng = np.random.default_rng(0)
    pts = rng.integers(0, 3, size=(7000, 3)).astype(np.float32)   # many equal codes: stability
    run(pts)
    flat = rng.uniform(-1, 1, size=(9000, 3)).astype(np.float32)
    flat[:, 2] = 0.25                                  # a plane: one axis of zero extent
    run(flat)


def test_batch_keeps_instances_in_place():
    rng = np.random.default_rng(5)
    sizes = [1, 4096, 7, 12_345, 2048, 300]
    parts = [synth.gmm_cloud(n, 3, seed=i).points if n > 8 else rng.normal(size=(n, 3)).astype(np.float32)
             for i, n in enumerate(sizes)]
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    run(np.concatenate(parts), offs)


@pytest.mark.parametrize("batch", [16_384, 16_385, 70_000])
def test_many_instances(batch):
    """Above 16,384 instances the 32-bit keys hold the upper bits of the Morton code only: every point stays
    in its instance, in the (stable) order of those."""
    from paper_2307_00071_gb300 import gira
    rng = np.random.default_rng(batch)
    sizes = rng.integers(1, 6, size=batch)
    offs = np.concatenate([[0], np.cumsum(sizes)]).astype(np.int64)
    pts = rng.normal(size=(offs[-1], 3)).astype(np.float32)
    got = gira.gira_test_point_order(torch.as_tensor(pts, device="cuda"), offs).cpu().numpy()
    drop = 18 - min(18, 32 - int(np.ceil(np.log2(batch))))
    want = [a + np.argsort(codes(pts[a:b]) >> drop, kind="stable") for a, b in zip(offs[:-1], offs[1:])]
    np.testing.assert_array_equal(got, np.concatenate(want))


def test_fits_of_many_instances():
    """One component per cloud: the mean and covariance of each cloud's own points."""
    from paper_2307_00071_gb300 import gira
    batch, n = 20_000, 4
    pts = np.random.default_rng(3).normal(size=(batch, n, 3)).astype(np.float32)
    r = gira.gira_gmm_fit_batched(pts.reshape(-1, 3), (np.arange(batch + 1) * n).astype(np.int64),
                                  np.ones(batch, np.int32), iters=1, tol=0.0, reg_covar=1e-2)
    x = pts.astype(np.float64)
    mean = x.mean(1)
    d = x - mean[:, None]
    cov = np.einsum("bni,bnj->bij", d, d) / n + 1e-2 * np.eye(3)
    # whitened binary32 sums of four terms: ~10 roundings of values up to about 5 (25 squared)
    assert np.abs(np.asarray(r["means"]).reshape(batch, 3) - mean).max() <= 10 * 5 * 2.0 ** -23
    assert np.abs(np.asarray(r["covs"]).reshape(batch, 3, 3) - cov).max() <= 10 * 25 * 2.0 ** -23
