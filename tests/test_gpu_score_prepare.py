"""What a given model needs before scoring (model_points_kernel: components of 32 per block, padding
slots and the points' packing in one launch) at the edges of its blocks, against the oracle within
the derived per-point bound; and which error is reported when several things are wrong."""
import numpy as np
import pytest

import oracle
from paper_2307_00071_gb300 import synth
from tests._parity import per_point_bound, to_np

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def gira():
    from paper_2307_00071_gb300 import gira as g
    return g


def model(k):
    cl = synth.gmm_cloud(4 * k + 300, min(k, 8), seed=k)
    rng = np.random.default_rng(k)
    means = cl.points[rng.choice(len(cl.points), k, replace=False)]
    covs = np.repeat((0.04 * np.eye(3))[None], k, 0)
    w = np.full(k, 1.0 / k)
    return cl.points, w.astype(np.float32), means.astype(np.float32), covs.astype(np.float32)


@pytest.mark.parametrize("n,k", [(1, 1), (255, 31), (256, 32), (257, 33), (1100, 257)])
@pytest.mark.parametrize("noalloc", [False, True])
def test_score_at_block_edges(gira, n, k, noalloc):
    import torch
    pts, w, mu, cov = model(k)
    pts = np.ascontiguousarray(pts[:n])
    args = [torch.as_tensor(a, device="cuda") for a in (pts, w, mu, cov)]
    call = gira.gira_gmm_loglik_noalloc if noalloc else gira.gira_gmm_loglik
    mean, pp = call(*args, per_point=True)
    _, _, ref = oracle.estep(pts, w, mu, cov, want_resp=False, want_lse=True)
    bound = per_point_bound(pts, w, mu, cov)
    assert np.all(np.abs(to_np(pp).astype(np.float64) - ref) <= bound)
    assert abs(mean - ref.mean()) <= np.mean(bound)


def test_a_non_finite_point_is_reported_before_a_bad_model(gira):
    pts, w, mu, cov = model(40)
    w, cov = w.copy(), cov.copy()
    w[3] = -1.0
    cov[20, 2, 2] = -1.0
    with pytest.raises(gira.GiraError) as e:
        gira.gira_gmm_loglik(pts, w, mu, cov)
    assert e.value.status != gira.ERR_NONFINITE_INPUT
    pts = pts.copy()
    pts[-1, 1] = np.nan
    for _ in range(20):
        with pytest.raises(gira.GiraError) as e:
            gira.gira_gmm_loglik(pts, w, mu, cov)
        assert e.value.status == gira.ERR_NONFINITE_INPUT
