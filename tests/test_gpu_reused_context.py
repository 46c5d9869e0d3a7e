"""A result does not depend on what the context computed before: bitwise the same on a fresh context and on one whose
buffers hold another problem.  Sizes at the lines of otgb_softmin's dispatch in one dimension (a small box of the columns
beside a sorted sweep) and above."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


@pytest.mark.parametrize("D,n,m", [(1, 61_100, 32_768), (1, 61_100, 32_769), (2, 61_100, 33_000), (3, 900, 800), (5, 700, 6000)])
def test_softmin_after_another_problem(D, n, m):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(D)
    q, p = T(rng.random((n, D), np.float32)), T(rng.random((m, D), np.float32))
    w, pot = T(np.full(m, 1.0 / m, np.float32)), T(0.01 * rng.normal(size=m).astype(np.float32))
    got = []
    for before in (None, (3.0, -0.5), (1e-3, 7.0)):
        ctx = otgb.Context()
        if before is not None:
            k = torch.full((n,), 1.0 / n, device="cuda")
            otgb.softmin(ctx, p, before[0] * q + before[1], k, 0.0 * k, 1.0)
            otgb.softmin(ctx, before[0] * q + before[1], before[0] * p[:50] + before[1], w[:50], pot[:50], 1.0)
        got.append(otgb.softmin(ctx, q, p, w, pot, 0.01))
        ctx.close()
    assert torch.equal(got[0], got[1]) and torch.equal(got[0], got[2])
