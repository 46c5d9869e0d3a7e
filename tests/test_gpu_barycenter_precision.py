"""The barycenter's gradient follows the precision of the solve: with OTGB_FP32_SIMT it is the CUDA-core sum over the kept
cluster pairs, with OTGB_FP32 the sum over every pair.  A truncation that drops pairs on purpose tells them apart."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


@pytest.mark.parametrize("precision", [0, 2])
def test_gradient_of_a_step_follows_the_precision(precision):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(1)
    n, m, blur = 900, 800, 1.5
    x, y = T(12.0 * rng.random((n, 3), np.float32)), T(12.0 * rng.random((m, 3), np.float32) + 0.5)
    a, b = T(np.full(n, 1.0 / n, np.float32)), T(np.full(m, 1.0 / m, np.float32))
    ctx = otgb.Context()
    p = otgb.default_params(blur=blur, reach=0.0, scaling=0.5, multiscale=1, cluster=0, cell=2.0, fixed_iters=10,
                            precision=precision, trunc_tau=0.5)
    r = otgb.sinkhorn_divergence(ctx, x, a, y, b, p, want_self=True)
    assert r["stats"]["kept_fraction"] < 0.7
    full = otgb.sinkhorn_grad_x(ctx, x, a, y, b, blur ** 2, r["f"], r["g"], r["a_self"])
    moved = x.clone()
    otgb.sinkhorn_barycenter(ctx, moved, a, [y], [b], p, iters=1, lr=1.0)
    step = (x - moved) * a[:, None]
    off = float((step - full).norm() / full.norm())
    assert (off < 1e-3) if precision == 0 else (off > 0.02), off
    ctx.close()
