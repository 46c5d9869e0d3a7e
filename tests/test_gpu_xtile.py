"""The tensor-core tiles against the FP64 oracle's softmin, at the edges of the tiles: point widths around the
K steps (4 .. 60 coordinates), sizes of one point, of a tile and one more, of less than a tile, of no multiple of
anything.  One coarse-to-fine step of the cluster-tiled form, and the dense sweep with its running shift."""
import numpy as np
import pytest
import torch

import oracle
from paper_2107_02010_gb300 import synth

pytestmark = pytest.mark.gpu
# the bars of the library: 1e-5 of the duals' scale in float32 (precision 0), 1e-3 in the reduced form (precision 1)
BAR = {0: 1e-5, 1: 1e-3}


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


@pytest.mark.parametrize("prec", [0, 1])
@pytest.mark.parametrize("D,n,m,K", [(4, 129, 257, 1), (5, 300, 260, 2), (12, 333, 290, 3), (13, 257, 128, 2),
                                     (16, 128, 129, 1), (28, 400, 301, 3), (29, 333, 290, 40), (44, 300, 517, 4),
                                     (45, 290, 333, 3), (60, 641, 500, 5), (60, 40, 37, 37), (60, 1, 200, 1)])
def test_one_step_matches_the_oracle(D, n, m, K, prec):
    from paper_2107_02010_gb300 import otgb

    if prec == 1 and D < 16:
        pytest.skip("the reduced-precision form needs D >= 16")
    x = synth.fiber_bundles(n, seed=4, perturb=3.0)[0][:, :D].copy()
    y = synth.fiber_bundles(m, seed=5)[0][:, :D].copy()
    rng = np.random.default_rng(6)
    a, b = (rng.uniform(0.5, 1.5, k).astype(np.float32) for k in (n, m))
    a, b = a / a.sum(), b / b.sum()
    b[0] = 0.0  # a column without weight
    blur, reach = 2.0, 20.0
    eps, lam = blur ** 2, 1.0 / (1.0 + blur ** 2 / reach ** 2)
    # duals near a solution: the row shift is an estimate of the result, not the result
    f, g, s, t = (np.zeros(k) for k in (n, m, n, m))
    for _ in range(3):
        f, g = oracle.softmin(x, y, b, g, eps, lam), oracle.softmin(y, x, a, f, eps, lam)
        s, t = 0.5 * (s + oracle.softmin(x, x, a, s, eps, lam)), 0.5 * (t + oracle.softmin(y, y, b, t, eps, lam))
    f, g, s, t = (v.astype(np.float32) for v in (f, g, s, t))
    want = {"f": 0.5 * (f + oracle.softmin(x, y, b, g.astype(np.float64), eps, lam)),
            "g": 0.5 * (g + oracle.softmin(y, x, a, f.astype(np.float64), eps, lam)),
            "a_self": 0.5 * (s + oracle.softmin(x, x, a, s.astype(np.float64), eps, lam)),
            "b_self": 0.5 * (t + oracle.softmin(y, y, b, t.astype(np.float64), eps, lam))}
    ctx = otgb.Context()
    dev = [T(v) for v in (f, g, s, t)]
    p = otgb.default_params(blur=blur, reach=reach, multiscale=1, cluster=1, k_clusters=K, precision=prec,
                            fixed_iters=1, max_iters=1, sigma_start=blur, translation=0, anderson=0,
                            f_init=dev[0].data_ptr(), g_init=dev[1].data_ptr(), a_init=dev[2].data_ptr(),
                            b_init=dev[3].data_ptr())
    out = otgb.sinkhorn_divergence(ctx, T(x), T(a), T(y), T(b), p, want_self=True)
    for k, w in want.items():
        err = np.max(np.abs(out[k].cpu().numpy() - w)) / (np.max(np.abs(w)) + eps)
        assert err < BAR[prec], (k, err)
    ctx.close()


@pytest.mark.parametrize("D,n,m", [(1, 129, 300), (2, 1, 40000), (3, 128, 1), (3, 4000, 2049), (3, 257, 128), (4, 1, 129), (5, 300, 1), (12, 129, 4000), (13, 257, 128), (16, 128, 127),
                                   (29, 130, 1025), (44, 64, 3001), (45, 290, 333), (60, 641, 2500), (60, 3000, 37)])
def test_dense_sweep_matches_the_oracle(D, n, m):
    from paper_2107_02010_gb300 import otgb

    q = synth.fiber_bundles(n, seed=4, perturb=3.0)[0][:, :D].copy()
    p = synth.fiber_bundles(m, seed=5)[0][:, :D].copy()
    rng = np.random.default_rng(7)
    w = rng.uniform(0.5, 1.5, m).astype(np.float32) / m
    if m > 1:
        w[rng.integers(0, m)] = 0.0
    eps, lam = 4.0, 1.0 / 1.01
    ctx = otgb.Context()
    # potentials of a few eps, and potentials that climb by 600 binades over the columns (the shift has to follow)
    for pot in (rng.normal(0.0, 12.0, m), np.linspace(-2000.0, 0.0, m)):
        pot = pot.astype(np.float32)
        old = rng.normal(0.0, 12.0, n).astype(np.float32)
        tilde = oracle.softmin(q, p, w, pot.astype(np.float64), eps, lam)
        for o, want in ((None, tilde), (old, 0.5 * (old + tilde))):
            got = otgb.softmin(ctx, T(q), T(p), T(w), T(pot), eps, lam=lam, old=None if o is None else T(o))
            err = np.max(np.abs(got.cpu().numpy() - want)) / (np.max(np.abs(want)) + eps)
            assert err < BAR[0], (err, o is None)
    # nothing but one column carries weight; and no finite answer where a potential is not finite
    w1 = np.zeros(m, np.float32)
    w1[m // 2] = 1.0
    want = oracle.softmin(q, p, w1, pot.astype(np.float64), eps, lam)
    got = otgb.softmin(ctx, T(q), T(p), T(w1), T(pot), eps, lam=lam).cpu().numpy()
    assert np.max(np.abs(got - want)) < BAR[0] * (np.max(np.abs(want)) + eps)
    pot[m // 2] = np.nan
    assert not np.any(np.isfinite(otgb.softmin(ctx, T(q), T(p), T(w1), T(pot), eps, lam=lam).cpu().numpy()))
    ctx.close()


@pytest.mark.parametrize("D,n,m,L,how", [(4, 1, 1, 1, "bundle"), (9, 129, 40, 3, "random"), (16, 200, 700, 20, "bundle"),
                                         (29, 300, 129, 5, "random"), (45, 131, 650, 40, "ignored"),
                                         (60, 1500, 1300, 20, "bundle"), (60, 257, 2000, 7, "random")])
def test_label_transfer_matches_the_oracle(D, n, m, L, how):
    """Labels along the bundles, labels that change from column to column, ignored labels, columns without weight, and
    rows so far away that they take the safe path."""
    from paper_2107_02010_gb300 import otgb

    x = synth.fiber_bundles(n, seed=4, perturb=3.0)[0][:, :D].copy()
    y, b, lab = synth.fiber_bundles(m, seed=5)
    y = y[:, :D].copy()
    rng = np.random.default_rng(8)
    if how != "bundle":
        lab = rng.integers(-1 if how == "ignored" else 0, L + (2 if how == "ignored" else 0), m).astype(np.int32)
    lab = lab.astype(np.int32)
    if m > 2:
        b[rng.integers(0, m)] = 0.0
    if n > 2:
        x[n // 2] += 40.0
    blur, eps, lam = 2.0, 4.0, 1.0 / 1.01
    a = np.full(n, 1.0 / n, np.float32)
    g = np.zeros(m)
    for _ in range(3):
        f = oracle.softmin(x, y, b, g, eps, lam)
        g = oracle.softmin(y, x, a, f, eps, lam)
    f, g = f.astype(np.float32), g.astype(np.float32)
    if n > 2:
        f[n // 2] = 0.0  # an outlier: its exponents are far below the float32 range
    ctx = otgb.Context()
    p = otgb.default_params(blur=blur, reach=20.0, fixed_iters=1)
    plan = otgb.sinkhorn_divergence(ctx, T(x), T(a), T(y), T(b), p, want_plan=True)["plan"]
    rsc, ram, rrm = oracle.transport_apply(x, y, b, eps, f.astype(np.float64), g.astype(np.float64), lab, L)
    for want_scores in (True, False):
        sc, am, rm = otgb.transport_apply(ctx, plan, T(f), T(g), T(lab), L, want_scores=want_scores)
        if want_scores:
            np.testing.assert_allclose(sc.cpu().numpy(), rsc, rtol=1e-4, atol=1e-5 * rsc.max())
        np.testing.assert_allclose(rm.cpu().numpy(), rrm, rtol=1e-4, atol=1e-30)
        top2 = np.sort(np.concatenate([rsc, np.zeros((n, 1))], axis=1), axis=1)[:, -2:]
        clear = (top2[:, 1] - top2[:, 0] >= 1e-4 * top2[:, 1]) & (rrm > 1e-30)
        assert np.all(am.cpu().numpy()[clear] == ram[clear])
    ctx.close()
