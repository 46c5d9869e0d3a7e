"""The sorted softmin where its blocks are loose and become one run: points on a line far longer than the blur, an outlier that
takes the resolution of the spatial order, potentials that make a run visit everything, rows that are no numbers among them.
Against FP64: no further off than the CUDA-core sweep, and by no more than 2e-3 eps (blocks of 16 units at s = 144: products of
5,000 rounded at 2^-24, and coordinates of 500 rounded at 3e-5 with a slope of s d = 7; a tile left out costs far more) but
beside the outlier, whose box centre of 50,000 rounds every coordinate at 4e-3 in both sweeps."""
import pytest
import torch

from test_gpu_not_slower import points
from test_gpu_softmin_error import softmin64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m,kind,eps,wild", [(46_001, 47_003, "line", 0.01, False), (33_001, 64_007, "line", 0.01, True),
                                               (46_001, 47_003, "outlier", 1.0, False), (64_007, 33_001, "outlier", 0.05, True),
                                               (46_001, 47_003, "cloud", 0.01, True)])
def test_loose_blocks(n, m, kind, eps, wild):
    from paper_2107_02010_gb300 import otgb

    g = torch.Generator(device="cuda").manual_seed(n)
    q, p = points(n, kind, g), points(m, kind, g)
    w = torch.rand(m, generator=g, device="cuda") + 0.5
    w /= w.sum()
    w[::50] = 0.0
    pot = (200.0 if wild else 1.0) * eps * torch.randn(m, generator=g, device="cuda")
    want = softmin64(q, p, w, pot, eps, 0.99)
    ctx = otgb.Context()
    got, cuda = otgb.softmin(ctx, q, p, w, pot, eps, 0.99), otgb.softmin_noalloc(q, p, w, pot, eps, 0.99)
    ok = torch.ones(n, dtype=torch.bool, device="cuda")
    if kind == "outlier":
        ok[7] = False  # its cost is 1e10: no digit of eps is left
    e, f = ((v.double() - want)[ok] for v in (got, cuda))
    assert e.square().mean() <= f.square().mean()
    if kind != "outlier":
        assert e.abs().max() <= 2e-3 * eps * (200.0 if wild else 1.0) ** 0.5
    # rows that are no numbers change no other row
    q2 = q.clone()
    q2[100::997] = float("nan")
    again = otgb.softmin(ctx, q2, p, w, pot, eps, 0.99)
    rest = ok & ~torch.isnan(q2[:, 0])
    assert torch.isfinite(again[rest]).all()
    if kind != "outlier":
        assert (again[rest] - got[rest]).abs().max() <= 4e-3 * eps * (200.0 if wild else 1.0) ** 0.5
    ctx.close()
