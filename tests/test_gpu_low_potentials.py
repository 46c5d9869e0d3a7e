"""One softmin sweep whose potentials are far beyond the costs: a mask value, or duals that drifted.  Every column has the same
potential v, so the result is -v to float32 accuracy; the terms' own exponents are as large as float32 holds, and what the
shift of a row is rounded by must not enter them."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("D,n,m", [(1, 1001, 803), (3, 1001, 803), (12, 1001, 803), (60, 130, 803), (63, 130, 803), (3, 46_001, 47_003)])
@pytest.mark.parametrize("v", [-1e9, -1e20, -1e30, 1e12, 1e30])
def test_result_is_minus_the_potential(D, n, m, v):
    from paper_2107_02010_gb300 import otgb

    g = torch.Generator(device="cuda").manual_seed(D)
    q, p = 10 * torch.rand(n, D, generator=g, device="cuda"), 10 * torch.rand(m, D, generator=g, device="cuda")
    w = torch.full((m,), 1.0 / m, device="cuda")
    pot = torch.full((m,), v, device="cuda")
    ctx = otgb.Context()
    for out in (otgb.softmin(ctx, q, p, w, pot, 0.5), otgb.softmin_noalloc(q, p, w, pot, 0.5)):
        # costs are at most 50 D = 3150 (3.2e-6 of 1e9); float32 rounding of an exponent and of the result 2e-7
        assert torch.allclose(out.double(), torch.full((n,), -v, device="cuda", dtype=torch.float64), rtol=4e-6, atol=0)
    ctx.close()
