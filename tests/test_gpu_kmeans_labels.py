"""Every label of the k-means indexes a cluster, also for points whose distances are no finite numbers: coordinates that are
not finite, and finite ones whose squares overflow.  Offsets and order are built from the labels, so a label out of range
would write past them."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,n,K", [(3, 300, 5), (60, 1000, 70), (61, 129, 1)])
def test_labels_of_points_without_a_finite_distance(D, n, K):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(D)
    x = rng.normal(size=(n, D)).astype(np.float32)
    init = rng.normal(size=(K, D)).astype(np.float32)
    odd = np.arange(0, n, 17)
    x[odd, 0] = np.resize(np.float32([np.nan, np.inf, -np.inf, 1e30, -3e38]), odd.size)
    ctx = otgb.Context()
    T = lambda v: torch.from_numpy(v).cuda()
    labels, _, perm, offsets = (v.cpu().numpy() for v in otgb.cluster_kmeans(ctx, T(x), K, iters=0, init=T(init)))
    assert labels.min() >= 0 and labels.max() < K
    assert np.array_equal(offsets, np.concatenate([[0], np.cumsum(np.bincount(labels, minlength=K))]))
    assert np.array_equal(perm, np.argsort(labels, kind="stable"))
    ok = np.setdiff1d(np.arange(n), odd)
    d = ((x[ok, None, :].astype(np.float64) - init[None].astype(np.float64)) ** 2).sum(-1)
    near = np.sort(d, axis=1)[:, :2] if K > 1 else np.c_[d, d + 1.0]
    clear = near[:, 1] - near[:, 0] > 1e-4 * near[:, 1]
    assert np.array_equal(labels[ok][clear], d.argmin(1)[clear])
    ctx.close()
