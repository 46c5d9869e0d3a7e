"""A device wait that gives up is never reported as success: the coarse phase of a coarse-to-fine solve,
and otgb_softmin in each of its forms (three dimensions, fiber vectors, one row block and split columns)."""
import numpy as np
import pytest
import torch

from paper_2107_02010_gb300 import synth

pytestmark = pytest.mark.gpu


def T(v):
    return torch.from_numpy(np.ascontiguousarray(v)).cuda()


@pytest.mark.parametrize("multiscale", [0, 1])
def test_a_wait_of_the_coarse_phase_reaches_the_caller(multiscale):
    from paper_2107_02010_gb300 import otgb

    x, a, y, b = (T(v) for v in synth.rotated_cloud(400, 360, seed=1))
    ctx = otgb.Context()
    kw = dict(blur=0.05, reach=0.5, multiscale=multiscale, cluster=0, cell=0.1)
    with pytest.raises(otgb.OtgbError) as e:
        otgb.sinkhorn_divergence(ctx, x, a, y, b, otgb.default_params(debug_wait_probe=2, **kw))
    assert e.value.code == -6
    out = otgb.sinkhorn_divergence(ctx, x, a, y, b, otgb.default_params(**kw))
    assert out["status"] == 0 and (out["stats"]["iters_coarse"] > 0) == bool(multiscale)
    ctx.close()


@pytest.mark.parametrize("D,n,m", [(3, 100, 90), (3, 300, 9000), (12, 300, 9000), (60, 130, 90), (64, 130, 90)])
def test_softmin_reports_a_wait_that_gave_up(D, n, m):
    from paper_2107_02010_gb300 import otgb

    rng = np.random.default_rng(D)
    q, p = T(rng.random((n, D), np.float32)), T(rng.random((m, D), np.float32))
    w, pot = T(np.full(m, 1.0 / m, np.float32)), T(np.zeros(m, np.float32))
    ctx = otgb.Context()
    want = otgb.softmin(ctx, q, p, w, pot, 0.1)
    ctx.debug_set(0, 1)
    with pytest.raises(otgb.OtgbError) as e:
        otgb.softmin(ctx, q, p, w, pot, 0.1)
    assert e.value.code == -6 and "wait" in str(e.value)
    ctx.debug_set(0, 0)
    assert torch.equal(otgb.softmin(ctx, q, p, w, pot, 0.1), want)
    ctx.close()
