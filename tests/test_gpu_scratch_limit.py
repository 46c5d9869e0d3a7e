"""Calls that can do with less scratch do so when an allocation fails (here: a limit on the bytes that a context may hold),
instead of returning ENOMEM: whatever the CUDA-core kernels can solve within a limit, the default forms solve too."""
import numpy as np
import pytest
import torch

from paper_2107_02010_gb300 import synth

pytestmark = pytest.mark.gpu
LIMIT = 1  # OTGB_DEBUG_SCRATCH_LIMIT


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


def under(limit, call):
    """call(context) on a fresh context that may hold `limit` bytes; None when it returns ENOMEM."""
    from paper_2107_02010_gb300 import otgb

    ctx = otgb.Context()
    ctx.debug_set(LIMIT, limit)
    try:
        return call(ctx)
    except otgb.OtgbError as e:
        assert e.code == -3, e
        return None
    finally:
        ctx.close()


def least(call):
    """The smallest limit within 3 % under which call succeeds."""
    lo, hi = 1, 1 << 33
    assert under(hi, call) is not None
    while hi > 1.03 * lo:
        mid = int((lo * hi) ** 0.5) if hi > 2 * lo else (lo + hi) // 2
        lo, hi = (lo, mid) if under(mid, call) is not None else (mid, hi)
    return hi


@pytest.mark.parametrize("multiscale", [0, 1])
def test_solve_within_the_scratch_of_the_cuda_core_form(multiscale):
    from paper_2107_02010_gb300 import otgb

    x, a, _ = synth.fiber_bundles(6000, seed=4, perturb=3.0)
    y, b, _ = synth.fiber_bundles(5000, seed=5)
    x, a, y, b = T(x), T(a), T(y), T(b)

    def solve(precision):
        p = otgb.default_params(blur=2.0, reach=20.0, multiscale=multiscale, cluster=1, k_clusters=40, fixed_iters=3,
                                precision=precision)
        return lambda ctx: otgb.sinkhorn_divergence(ctx, x, a, y, b, p)

    limit = least(solve(2))
    want = under(1 << 33, solve(2))
    for room in (1.0, 1.05, 1.2, 1.5, 3.0):
        got = under(int(room * limit), solve(0))
        assert got is not None, room
        assert abs(got["S"] - want["S"]) <= 1e-5 * abs(want["S"])
    # a context that once failed goes on working
    ctx = otgb.Context()
    ctx.debug_set(LIMIT, limit // 4)
    with pytest.raises(otgb.OtgbError) as e:
        solve(0)(ctx)
    assert e.value.code == -3
    ctx.debug_set(LIMIT, 0)
    assert abs(solve(0)(ctx)["S"] - want["S"]) <= 1e-5 * abs(want["S"])
    ctx.close()


def test_label_transfer_within_the_scratch_of_the_cuda_core_form():
    from paper_2107_02010_gb300 import otgb

    n, m, L = 6000, 5000, 30
    x, a, _ = synth.fiber_bundles(n, seed=4, perturb=3.0)
    y, b, lab = synth.fiber_bundles(m, seed=5)
    a, b, lab = T(a), T(b), T((lab % L).astype(np.int32))
    ctx = otgb.Context()
    p = otgb.default_params(blur=2.0, reach=20.0, multiscale=1, cluster=1, k_clusters=20, fixed_iters=5)

    def transfer(pad):  # 64 coordinates (the last ones 0) take the CUDA-core kernel
        X, Y = (T(np.pad(v, ((0, 0), (0, pad)))) for v in (x, y))
        r = otgb.sinkhorn_divergence(ctx, X, a, Y, b, p, want_plan=True)
        return lambda c: otgb.transport_apply(c, r["plan"], r["f"], r["g"], lab, L, want_scores=False)

    general, call = transfer(4), transfer(0)
    limit = least(general)
    _, am, rm = under(1 << 33, general)
    for room in (1.0, 1.05, 1.2, 1.5, 3.0):
        got = under(int(room * limit), call)
        assert got is not None, room
        assert (got[1] != am).float().mean() < 1e-3
        assert torch.allclose(got[2], rm, rtol=1e-3)
    ctx.close()


@pytest.mark.parametrize("D,n,m", [(3, 50_000, 45_000), (60, 300, 20_000)])
def test_softmin_within_the_scratch_of_a_plain_sweep(D, n, m):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(3)
    q, p = (T(10.0 * rng.random((k, D), np.float32)) for k in (n, m))
    w, pot = T(np.full(m, 1.0 / m, np.float32)), T(rng.normal(size=m).astype(np.float32))
    call = lambda ctx: otgb.softmin(ctx, q, p, w, pot, 0.5)
    want = under(1 << 33, call)
    # packed rows and columns with their log weights, a list entry per row, and 150 KB of small buffers
    limit = 4 * ((D + 3) & ~3) * (n + m) + 16 * (n + 64) + (4 * m if D > 3 else 0) + 150_000
    got = under(limit, call)
    assert got is not None
    assert (got - want).abs().max() <= 1e-5 * (want.abs().max() + 0.5)


def test_gradient_within_no_scratch():
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(4)
    n, m = 9000, 8000
    x, y = (T(10.0 * rng.random((k, 3), np.float32)) for k in (n, m))
    a, b = (T(np.full(k, 1.0 / k, np.float32)) for k in (n, m))
    f, g = (T(rng.normal(size=k).astype(np.float32)) for k in (n, m))
    call = lambda ctx: otgb.sinkhorn_grad_x(ctx, x, a, y, b, 0.5, f, g, f)
    want, got = under(1 << 33, call), under(4096, call)
    assert got is not None
    assert (got - want).abs().max() <= 1e-5 * want.abs().max()
