"""Forms chosen by a rule on sizes are not slower than the general form where the data are not what they were made for: blocks
that are loose at the blur, an outlier that takes the resolution of the spatial order, points on a line.  Times are the best
of five calls; the bar is 1.3 times the general form's (the faults it is for took 1.5 to 20 times)."""
import time

import pytest
import torch

pytestmark = pytest.mark.gpu


def best(fn, reps=5):
    fn()
    fn()
    out = []
    for _ in range(reps):
        torch.cuda.synchronize()
        t = time.perf_counter()
        fn()
        torch.cuda.synchronize()
        out.append(time.perf_counter() - t)
    return min(out)


def points(n, kind, g):
    x = 30.0 * torch.rand(n, 3, generator=g, device="cuda")
    if kind == "outlier":
        x[7] = 1e5
    if kind == "line":
        x = torch.cat([1000.0 * torch.rand(n, 1, generator=g, device="cuda"), torch.zeros(n, 2, device="cuda")], 1)
    return x


@pytest.mark.parametrize("n,m,kind,eps", [(1400, 4400, "cloud", 0.05), (2000, 2000, "cloud", 1.0), (3000, 3000, "cloud", 0.05),
                                          (20_000, 20_000, "outlier", 1.0), (20_000, 20_000, "line", 0.01)])
def test_gradient(n, m, kind, eps):
    from paper_2107_02010_gb300 import otgb

    g = torch.Generator(device="cuda").manual_seed(1)
    x, y = points(n, kind, g), points(m, kind, g)
    a, b = torch.full((n,), 1.0 / n, device="cuda"), torch.full((m,), 1.0 / m, device="cuda")
    f, h = torch.zeros(n, device="cuda"), torch.zeros(m, device="cuda")
    ctx = otgb.Context()
    t = [best(lambda: otgb.sinkhorn_grad_x(ctx, u, a, v, b, eps, f, h, f))
         for u, v in ((x, y), tuple(torch.nn.functional.pad(w, (0, 1)).contiguous() for w in (x, y)))]  # 4-D: every pair
    ctx.close()
    assert t[0] <= 1.3 * t[1], t


@pytest.mark.parametrize("n,kind,eps,wild", [(46_000, "cloud", 0.01, True), (100_000, "line", 0.01, False), (46_000, "line", 0.01, True),
                                             (46_000, "outlier", 1.0, False), (46_000, "outlier", 0.05, False)])
def test_softmin(n, kind, eps, wild):
    from paper_2107_02010_gb300 import otgb

    g = torch.Generator(device="cuda").manual_seed(2)
    q, p = points(n, kind, g), points(n, kind, g)
    w, pot = torch.full((n,), 1.0 / n, device="cuda"), torch.zeros(n, device="cuda")
    if wild:  # potentials that reach far beyond the neighbours
        pot = 200.0 * eps * torch.randn(n, generator=g, device="cuda")
    ctx = otgb.Context()
    t = best(lambda: otgb.softmin(ctx, q, p, w, pot, eps)), best(lambda: otgb.softmin_noalloc(q, p, w, pot, eps))
    ctx.close()
    assert t[0] <= 1.3 * t[1], t
