"""otgb_softmin with a few points very far from all others, so that a block's centre is far from its rows: what the products of
the dot-product form are rounded by is then larger than any exponent, and a row must not keep it.  Against FP64.  The packed
coordinates are relative to the middle of the columns' box: with a far column they are rounded to 2^-25 of its distance F, which
moves the cost of a pair by up to 2 x 2^-25 F |x - y|_1."""
import pytest
import torch

from test_gpu_softmin_error import softmin64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", ["rows", "rows and columns"])
@pytest.mark.parametrize("D,n,m,far", [(1, 700, 650, 1e5), (2, 130, 3000, 3e5), (3, 700, 650, 1e5), (3, 3000, 129, 1e6), (12, 700, 650, 1e6),
                                       (60, 300, 650, 1e6), (3, 46_001, 47_003, 1e6)])
def test_far_rows(D, n, m, far, which):
    from paper_2107_02010_gb300 import otgb

    g = torch.Generator(device="cuda").manual_seed(D + n)
    q = 4 / D**0.5 * torch.rand(n, D, generator=g, device="cuda")
    p = 4 / D**0.5 * torch.rand(m, D, generator=g, device="cuda")
    w = torch.full((m,), 1.0 / m, device="cuda")
    pot = 0.3 * torch.rand(m, generator=g, device="cuda")
    q[:: n // 2] = far
    if which != "rows":
        p[m // 3] = far
    eps = 0.09
    ctx = otgb.Context()
    for out in (otgb.softmin(ctx, q, p, w, pot, eps), otgb.softmin(ctx, q, p, w, pot, eps, 0.97, q[:, 0].contiguous() * 0, 1.0) / 0.97):
        want = softmin64(q, p, w, pot, eps, 1.0)
        # near rows without a far column: 1e-5, as in every other test of the sweep; |x - y|_1 <= 4 sqrt(D)
        atol = 1e-5 if which == "rows" else 2 * 2.0**-25 * far * 4 * D**0.5
        assert ((out.double() - want).abs() <= atol + 2e-6 * want.abs()).all()
    ctx.close()
