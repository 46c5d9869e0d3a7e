"""The sorted 3-D sums (large otgb_softmin, sinkhorn_grad_x for D <= 3) against the FP64 oracle: sizes that are no
multiple of a tile, one and two dimensions, clouds with far outliers and columns without weight, potentials whose best
column lies far from the row, and duals that are far from a solution."""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu
TOL = 1e-5  # the library's float32 bar


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


def cloud(rng, n, D, scale):
    x = rng.uniform(0.0, scale, size=(n, D)).astype(np.float32)
    x[:: max(1, n // 7)] += 5.0 * scale  # outliers
    return x


@pytest.mark.parametrize("D,n,m,how", [(3, 45_001, 44_999, "near"), (3, 4097, 500_000, "ramp"), (2, 60_000, 40_000, "near"),
                                       (1, 50_000, 45_000, "ramp"), (3, 4096, 530_000, "near"), (3, 32_768, 530_000, "ramp")])
def test_large_softmin_sampled_rows(D, n, m, how):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(n)
    q, p = cloud(rng, n, D, 30.0), cloud(rng, m, D, 30.0)
    w = rng.uniform(0.5, 1.5, m).astype(np.float32) / m
    w[rng.integers(0, m, 100)] = 0.0
    eps, lam = 1.0, 1.0 / 1.01
    pot = rng.normal(0.0, 3.0, m)
    if how == "ramp":
        pot += 20.0 * p[:, 0]  # the best column is 20 units away along the first axis
    pot = pot.astype(np.float32)
    old = rng.normal(0.0, 3.0, n).astype(np.float32)
    ctx = otgb.Context()
    idx = np.unique(np.concatenate([np.arange(0, n, max(1, n // 7)), rng.integers(0, n, 100), [n - 1]]))
    tilde = oracle.softmin(q[idx], p, w, pot.astype(np.float64), eps, lam)
    for o in (None, old):
        got = otgb.softmin(ctx, T(q), T(p), T(w), T(pot), eps, lam=lam, old=None if o is None else T(o)).cpu().numpy()
        assert np.all(np.isfinite(got))
        want = tilde if o is None else 0.5 * (old[idx] + tilde)
        assert np.max(np.abs(got[idx] - want)) < TOL * (np.max(np.abs(want)) + eps)
    ctx.close()


@pytest.mark.parametrize("D,n,m,shift", [(3, 5003, 4100, 0.0), (2, 4400, 777, 0.0), (1, 4500, 129, 0.0), (3, 4471, 3000, 30.0),
                                         (3, 2000, 2001, 0.0)])
def test_gradient_matches_oracle(D, n, m, shift):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(n + D)
    x, y = cloud(rng, n, D, 20.0), cloud(rng, m, D, 20.0)
    a, b = (rng.uniform(0.5, 1.5, k).astype(np.float32) for k in (n, m))
    a, b = a / a.sum(), b / b.sum()
    a[3] = b[5] = 0.0
    eps, lam = 1.0, 1.0 / 1.01
    f, g, s = np.zeros(n), np.zeros(m), np.zeros(n)
    for _ in range(2):
        f = oracle.softmin(x, y, b, g, eps, lam)
        g = oracle.softmin(y, x, a, f, eps, lam)
        s = 0.5 * (s + oracle.softmin(x, x, a, s, eps, lam))
    f, g, s = (f - shift).astype(np.float32), g.astype(np.float32), (s - 0.5 * shift).astype(np.float32)
    ctx = otgb.Context()
    got = otgb.sinkhorn_grad_x(ctx, T(x), T(a), T(y), T(b), eps, T(f), T(g), T(s)).cpu().numpy()
    want = oracle.grad_x(x, a, y, b, eps, s.astype(np.float64), f.astype(np.float64), g.astype(np.float64))
    assert np.max(np.abs(got - want)) < TOL * np.max(np.abs(want))
    ctx.close()
