"""The tensor-core sweeps are no further from FP64 than the CUDA-core sweep of the same problem (otgb_softmin_noalloc): the
rms error over all rows, for clouds whose blocks of rows span the whole domain."""
import numpy as np
import pytest
import torch

from paper_2107_02010_gb300 import synth

pytestmark = pytest.mark.gpu


def softmin64(q, p, w, pot, eps, lam):
    q, p, pot, lw = q.double(), p.double(), pot.double(), torch.log(w.double())
    c = p.mean(0)
    q, p = q - c, p - c
    h = lw + (pot - 0.5 * (p * p).sum(1)) / eps
    out = [-lam * (eps * torch.logsumexp(h + (u @ p.T) / eps, 1) - 0.5 * (u * u).sum(1)) for u in q.split(1000)]
    return torch.cat(out)


def errors(n, m, D, side, eps, seed, cloud):
    from paper_2107_02010_gb300 import otgb

    g = torch.Generator(device="cuda").manual_seed(seed)
    q, p = cloud(n, D, side, g), cloud(m, D, side, g)
    w = torch.rand(m, generator=g, device="cuda") + 0.5
    w /= w.sum()
    pot = 3.0 * eps * torch.randn(m, generator=g, device="cuda")
    want = softmin64(q, p, w, pot, eps, 0.99)
    ctx = otgb.Context()
    got = otgb.softmin(ctx, q, p, w, pot, eps, 0.99), otgb.softmin_noalloc(q, p, w, pot, eps, 0.99)
    ctx.close()
    return [float((v.double() - want).square().mean().sqrt()) for v in got]


def uniform(n, D, side, g):
    return side * torch.rand(n, D, generator=g, device="cuda")


@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("n,m,side,eps", [(3000, 2500, 30.0, 1.0), (500, 60_000, 30.0, 1.0), (3000, 2500, 1.0, 0.0025)])
def test_dense_sweep_in_up_to_three_dimensions(D, n, m, side, eps):
    e = [errors(n, m, D, side, eps, seed, uniform) for seed in range(3)]
    tc, cuda = (sum(v[k] ** 2 for v in e) ** 0.5 for k in (0, 1))
    assert tc <= cuda, (tc, cuda)


@pytest.mark.parametrize("D", [1, 2, 3])
@pytest.mark.parametrize("side,eps", [(30.0, 1.0), (1.0, 0.0025)])
def test_sorted_sweep(D, side, eps):
    """Thousands of columns in a row's sum, most of them small beside it."""
    e = [errors(46_001, 47_003, D, side, eps, seed, uniform) for seed in range(2)]
    tc, cuda = (sum(v[k] ** 2 for v in e) ** 0.5 for k in (0, 1))
    assert tc <= cuda, (tc, cuda)


def fibers(n, D, side, g):
    x = synth.fiber_bundles(n, seed=int(torch.randint(0, 1 << 30, (1,), generator=g, device="cuda")), perturb=3.0)[0]
    return torch.from_numpy(np.ascontiguousarray(x[:, :D])).cuda()


@pytest.mark.parametrize("D,cloud,eps", [(4, uniform, 1.0), (7, uniform, 4.0), (12, uniform, 25.0), (4, fibers, 25.0), (5, fibers, 25.0),
                                         (13, fibers, 4.0), (24, fibers, 4.0), (45, fibers, 1.0), (60, fibers, 4.0)])
def test_dense_sweep_in_more_dimensions(D, cloud, eps):
    e = [errors(3001, 2777, D, 30.0, eps, seed, cloud) for seed in range(3)]
    tc, cuda = (sum(v[k] ** 2 for v in e) ** 0.5 for k in (0, 1))
    assert tc <= cuda, (tc, cuda)


def solve64(x, a, y, b, blur, reach, steps):
    """The averaged loop with its schedule and the translation of (f, g), in FP64."""
    box = torch.cat([x, y]).double()
    d = float((box.amax(0) - box.amin(0)).square().sum().sqrt())
    sched = []
    while d > blur:
        sched.append(d)
        d *= 0.5
    f, g = torch.zeros_like(a, dtype=torch.float64), torch.zeros_like(b, dtype=torch.float64)
    rho = reach * reach
    for sigma in sched + [blur] * (steps + 1):
        eps = sigma * sigma
        lam = 1.0 / (1.0 + eps / rho)
        f2, g2 = softmin64(x, y, b, g, eps, lam), softmin64(y, x, a, f, eps, lam)
        f, g = 0.5 * (f + f2), 0.5 * (g + g2)
        c = 0.5 * rho * torch.log((a * torch.exp(-f / rho)).sum() / (b * torch.exp(-g / rho)).sum())
        f, g = f + c, g - c
    return f, g


def test_the_schedule_leaves_no_bias_in_the_slow_modes():
    """After the schedule and ten steps f and g hold what every step left in the translations of the bundles (they contract
    by less than 1 % per step), so that a loss of the same sign in every step adds up.  Error of the single-scale float32 solve
    over that of its CUDA-core form, geometric mean over twenty problems: no larger than 1, within the 11 % that the spread
    between problems (a factor of 1.6) leaves to the mean."""
    from paper_2107_02010_gb300 import otgb

    ratio = 1.0
    for P in (16, 20):
        for seed in range(10):
            x, y = (torch.from_numpy(synth.fiber_bundles(n, seed=q + seed, P=P, perturb=3.0)[0]).cuda()
                    for n, q in ((1500, 100), (1300, 200)))
            a, b = (torch.full((len(v),), 1.0 / len(v), device="cuda") for v in (x, y))
            want = solve64(x, a, y, b, 2.0, 20.0, 10)
            err = []
            for precision in (0, 2):
                ctx = otgb.Context()
                p = otgb.default_params(blur=2.0, reach=20.0, scaling=0.5, fixed_iters=10, precision=precision)
                r = otgb.sinkhorn_divergence(ctx, x, a, y, b, p)
                err.append(sum(float((r[k].double() - w).square().sum()) for k, w in zip(("f", "g"), want)) ** 0.5)
                ctx.close()
            assert err[0] < 1e-5 * float(want[0].norm())
            ratio *= (err[0] / err[1]) ** 0.05
    assert ratio <= 1.11, ratio
