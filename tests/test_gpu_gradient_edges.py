"""The gradient over sorted points against the form that sums every pair (the same points with a fourth coordinate 0), for
inputs at which a skipped tile or an early exit would show: columns without weight that are no numbers, rows that are no
numbers, a potential that is not finite, points that coincide, weights in a single column."""
import pytest
import torch

pytestmark = pytest.mark.gpu


def both(n, m, change, side=10.0):
    from paper_2107_02010_gb300 import otgb

    g = torch.Generator(device="cuda").manual_seed(n)
    x, y = side * torch.rand(n, 3, generator=g, device="cuda"), side * torch.rand(m, 3, generator=g, device="cuda")
    a, b = torch.rand(n, generator=g, device="cuda") + 0.5, torch.rand(m, generator=g, device="cuda") + 0.5
    f, h = torch.randn(n, generator=g, device="cuda"), torch.randn(m, generator=g, device="cuda")
    v = dict(x=x, y=y, a=a / a.sum(), b=b / b.sum(), f=f - 3.0, h=h, s=-3.0 + 0.1 * f)
    change(v)
    ctx = otgb.Context()
    out = []
    for pad in (0, 1):
        X, Y = (torch.nn.functional.pad(v[k], (0, pad)).contiguous() for k in "xy")
        out.append(otgb.sinkhorn_grad_x(ctx, X, v["a"], Y, v["b"], 0.5, v["f"], v["h"], v["s"])[:, :3])
    ctx.close()
    return out


def dead_columns(v):
    v["b"][::9] = 0.0
    v["y"][::27] = float("nan")  # without weight: no term


def bad_rows(v):
    v["a"][5::700] = 0.0
    v["x"][5::700] = float("nan")
    v["f"][11] = float("nan")
    v["f"][12] = float("inf")
    v["f"][13] = -float("inf")


def bad_potential(v):
    v["h"][17] = float("nan")


def coincident(v):
    v["x"][:] = v["x"][:1]
    v["y"][: len(v["y"]) // 2] = v["x"][0]


def one_column(v):
    v["b"][:] = 0.0
    v["b"][len(v["b"]) // 2] = 1.0


@pytest.mark.parametrize("n,m", [(2830, 1), (2001, 2049), (257, 40_000)])
@pytest.mark.parametrize("change", [dead_columns, bad_rows, bad_potential, coincident, one_column])
def test_sorted_gradient_is_that_of_every_pair(n, m, change):
    if m == 1 and change in (dead_columns, bad_potential):
        pytest.skip("needs more than one column")
    got, want = both(n, m, change)
    assert torch.equal(torch.isnan(got), torch.isnan(want))
    ok = torch.isfinite(want)
    assert (got[ok] - want[ok]).abs().max() <= 1e-5 * want[ok].abs().max() if ok.any() else True
