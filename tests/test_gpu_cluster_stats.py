"""Cluster masses, centroids and spreads of points in more than three dimensions when the sums leave the range in which float
products keep their error terms: the cluster scale of a solve does not depend on the size of the weights."""
import numpy as np
import pytest
import torch

from paper_2107_02010_gb300 import synth

pytestmark = pytest.mark.gpu


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


@pytest.mark.parametrize("D", [5, 36, 64])
def test_cluster_scale_does_not_depend_on_the_size_of_the_weights(D):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(D)
    x, y = (rng.normal(size=(n, D)).astype(np.float32) + 5.0 * rng.integers(0, 4, (n, 1)).astype(np.float32) for n in (700, 650))
    a, b = (rng.uniform(0.5, 1.5, n).astype(np.float32) for n in (700, 650))
    a[3] = b[5] = 0.0
    got = []
    for scale in (1.0, 2.0 ** -96, 2.0 ** 60):
        ctx = otgb.Context()
        p = otgb.default_params(blur=1.0, multiscale=1, cluster=1, k_clusters=9, fixed_iters=1, precision=2)
        r = otgb.sinkhorn_divergence(ctx, T(x), T(a * np.float32(scale)), T(y), T(b * np.float32(scale)), p, raise_on_noconv=False)
        got.append(r["stats"]["sigma_switch"])
        ctx.close()
    # two float roundings of a mean of squares, under a square root
    assert np.allclose(got[1:], got[0], rtol=2.0 ** -22), got
