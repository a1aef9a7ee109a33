"""Tensor-core products on CTA pairs (K >= 512, at most a quarter of a tile's columns padding) and on single CTAs beside
them: Theta and the adjoint against the CPU FP64 oracle, at one column tile and at ragged ones, with ragged row blocks."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2208_07731_gb300 as isdf
from paper_2208_07731_gb300 import workload as W

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
THETA_TOL, GRAD_TOL = 1e-5, 1e-4   # the mode's bounds


# n_orb = 256 has K = 512 in the Gram product; 2 n_mu columns: 128 (single CTAs), 256 (one tile), 384 (a quarter padding),
# 640 (two tiles and a half); n_orb = 32 keeps the Gram on single CTAs beside a fit on pairs
@pytest.mark.parametrize("n_orb,n_mu,max_rows", [(256, 64, 777), (256, 128, 1000), (256, 192, 4096), (256, 320, 1033),
                                                 (32, 256, 255)])
def test_pairs_against_oracle(n_orb, n_mu, max_rows):
    w = W.Workload("pairs", 20, 10.0, n_orb, n_mu, "c64", 0, 10.0, (0.25, 0.0, 0.0), "none", 40)
    phi, psi = (x.to(torch.complex64) for x in W.make_pair(w))
    idx = np.random.default_rng(n_mu).permutation(20 ** 3)[:n_mu].astype(np.int64)
    plan = isdf.Plan(phi.to(DEV), psi.to(DEV), torch.from_numpy(idx), mode="mixed", max_rows=max_rows)
    theta = plan.fit_theta(101, 3001).cpu().numpy().astype(np.complex128)
    K = W.loss_matrix(n_mu, 5)
    _, gphi, gpsi = isdf.surrogate_loss_and_grad(plan, torch.from_numpy(K).to(DEV), w.dV)
    plan.check()
    p64, q64 = phi.numpy(), psi.numpy()
    full = O.fit_theta(p64, q64, idx)["theta"]
    assert np.linalg.norm(theta - full[101:3102]) < THETA_TOL * np.linalg.norm(full[101:3102])
    ref = O.theta_backward(p64, q64, idx, lambda rows, T: O.surrogate_grad_theta(T, K, w.dV))
    for got, exp in ((gphi, ref["grad_phi"]), (gpsi, ref["grad_psi"])):
        assert np.linalg.norm(got.cpu().numpy() - exp) < GRAD_TOL * np.linalg.norm(exp)


def test_launches_of_a_block_agree():
    """A row block longer than a launch (65,536 rows at N_mu = 1024) and blocks shorter than one: identical Theta."""
    g = torch.Generator(device=DEV).manual_seed(7)
    phi, psi = (torch.randn(70001, 32, dtype=torch.complex64, device=DEV, generator=g) for _ in range(2))
    idx = torch.randperm(70001, device=DEV, generator=g)[:1024].sort().values
    long, short = (isdf.Plan(phi, psi, idx, mode="mixed", max_rows=m) for m in (70001, 30001))
    a, b = long.fit_theta(), short.fit_theta()
    long.check(), short.check()
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))


@pytest.mark.parametrize("n_orb,n_mu", [(256, 128), (256, 320), (32, 256)])
def test_loss_of_products_on_pairs(n_orb, n_mu):
    """The surrogate loss is quadratic in Theta: twice Theta's bound."""
    w = W.Workload("pairs", 20, 10.0, n_orb, n_mu, "c64", 0, 10.0, (0.25, 0.0, 0.0), "none", 40)
    phi, psi = (x.to(torch.complex64) for x in W.make_pair(w))
    idx = np.random.default_rng(n_mu).permutation(20 ** 3)[:n_mu].astype(np.int64)
    plan = isdf.Plan(phi.to(DEV), psi.to(DEV), torch.from_numpy(idx), mode="mixed", max_rows=1000)
    K = W.loss_matrix(n_mu, 5)
    loss, _, _ = isdf.surrogate_loss_and_grad(plan, torch.from_numpy(K).to(DEV), w.dV)
    plan.check()
    T = O.fit_theta(phi.numpy(), psi.numpy(), idx)["theta"]
    ref = w.dV * float(np.sum((T.conj() * (T @ K.T)).real))
    assert abs(float(loss) - ref) < 2 * THETA_TOL * abs(ref)


def test_wait_that_runs_out_in_the_gram_product():
    """The Gram product on pairs takes its time-out path (the MMA issuer waits 20,000 cycles on a barrier that nothing
    signals): reported, and the same plan fits as before after an update."""
    g = torch.Generator(device=DEV).manual_seed(9)
    phi, psi = (torch.randn(2000, 256, dtype=torch.complex64, device=DEV, generator=g) for _ in range(2))
    idx = torch.randperm(2000, device=DEV, generator=g)[:256].sort().values
    plan = isdf.Plan(phi, psi, idx, mode="mixed", max_rows=2000)
    ref = plan.fit_theta()
    plan.check()
    plan.set_wait_budget(-20000)
    plan.fit_theta()
    assert plan.status()[0] == 6
    plan.set_wait_budget(0)
    plan.update(idx)
    assert torch.equal(torch.view_as_real(plan.fit_theta()), torch.view_as_real(ref))
    plan.check()
