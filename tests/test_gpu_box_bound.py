"""Truncation by the distance of the clusters' bounding boxes (cold coarse-to-fine solves, D <= 3) in one and two dimensions
and for p = 1, against the converged FP64 oracle, at the settings and the bar of the three-dimensional parity test (blur 1.5,
reach 4: well-conditioned duals, so the library's float32 bar of 1e-5 holds whatever was kept)."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
TOL = 1e-5


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


@pytest.mark.parametrize("D,p,side,cell", [(1, 2, 60.0, 2.0), (2, 2, 30.0, 2.0), (2, 2, 30.0, 0.4), (3, 1, 12.0, 3.0)])
def test_box_truncation_matches_oracle(D, p, side, cell):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(D)
    n, m, blur, reach = 1203, 901, 1.5, 4.0
    x = (side * rng.random((n, D))).astype(np.float32)
    y = (side * rng.random((m, D)) + 1.0).astype(np.float32)
    a, b = (rng.uniform(0.5, 1.5, k).astype(np.float32) for k in (n, m))
    a[7] = b[9] = 0.0
    a, b = a / a.sum(), b / b.sum()
    ref = oracle.sinkhorn(x, a, y, b, blur=blur, reach=reach, scaling=0.5, p=p, tol=1e-12, max_iters=20000)
    assert ref["converged"]
    ctx = otgb.Context()
    out = otgb.sinkhorn_divergence(ctx, T(x), T(a), T(y), T(b), otgb.default_params(
        p=p, blur=blur, reach=reach, scaling=0.5, multiscale=1, cluster=0, cell=cell, tol=1e-8), want_self=True)
    assert out["stats"]["kept_fraction"] < 0.9 or p == 1
    assert abs(out["S"] - ref["S"]) <= TOL * abs(ref["S"]), (out["S"], ref["S"])
    for k, key in (("f", "f"), ("g", "g"), ("a_self", "a"), ("b_self", "b")):
        got = out[k].cpu().numpy().astype(np.float64)
        assert np.max(np.abs(got - ref[key])) < TOL * (np.max(np.abs(ref[key])) + blur ** p), k
    ctx.close()
