"""A matrix M that is not positive definite, found while many CTAs of a Cholesky step are at work and other plans update on
streams of their own: every plan reports its own pivot, and a later update with independent points fits as a fresh plan."""
import pytest
import torch

import paper_2208_07731_gb300 as isdf

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("n,n_mu", [(32, 192), (64, 640)])
def test_plans_on_streams_report_their_pivots(n, n_mu):
    g = torch.Generator(device=DEV).manual_seed(n_mu)
    n_r = 2 * n_mu
    phi, psi = (torch.randn(n_r, n, dtype=torch.complex128, device=DEV, generator=g) for _ in range(2))
    good = torch.arange(n_mu, device=DEV)
    # the second of two equal points leaves a pivot of rounding size: in the first block, at a block's first and last column,
    # in the last block, and none
    bad = [3, 16, 47, n_mu // 2 + 5, n_mu - 1, None]
    points = []
    for b in bad:
        idx = good.clone()
        if b is not None:
            idx[b] = idx[b // 2]
        points.append(idx)
    plans = [isdf.Plan(phi, psi, good, mode="mixed", max_rows=n_r) for _ in bad]
    ref = plans[0].fit_theta()
    streams = [torch.cuda.Stream() for _ in bad]
    torch.cuda.synchronize()
    for _ in range(8):
        for plan, idx, st in zip(plans, points, streams):
            plan.update(idx, stream=st)
        assert [plan.status() for plan in plans] == [(0, 0) if b is None else (3, b) for b in bad]
    for plan in plans:
        plan.update(good)
        assert torch.equal(torch.view_as_real(plan.fit_theta()), torch.view_as_real(ref))
        plan.check()
