"""FP64 adjoint: every row block takes the exact-slicing products whatever its length and the plan's sizes, so the
gradients do not depend on the row blocks that the plan was made for."""
import pytest
import torch

import paper_2208_07731_gb300 as isdf

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _grads(phi, psi, idx, rows, max_rows, g):
    plan = isdf.Plan(phi, psi, idx, mode="fp64", max_rows=max_rows)
    a, b = (torch.zeros(phi.shape, dtype=torch.complex128, device=DEV) for _ in range(2))
    plan.backward(rows[0], rows[1], a, b, grad_theta=g)
    torch.cuda.synchronize()
    n = isdf.kernel_launches()
    plan.backward(rows[0], rows[1], a, b, grad_theta=g)
    n = isdf.kernel_launches() - n
    plan.backward_finalize(a, b)
    plan.check()
    return torch.view_as_real(a), torch.view_as_real(b), n


def test_a_ragged_block_with_longer_slabs():
    """Blocks of 14,400 rows are sliced in slabs of 4,800; the last one, of 7,000, is one slab."""
    gen = torch.Generator(device=DEV).manual_seed(1)
    phi, psi = (torch.randn(21400, 48, dtype=torch.complex128, device=DEV, generator=gen) for _ in range(2))
    idx = torch.randperm(21400, device=DEV, generator=gen)[:96].sort().values
    g = torch.randn(7000, 96, dtype=torch.complex128, device=DEV, generator=gen)
    long, exact = (_grads(phi, psi, idx, (14400, 7000), m, g) for m in (14400, 7000))
    assert torch.equal(long[0], exact[0]) and torch.equal(long[1], exact[1]) and long[2] == exact[2]


def test_more_orbitals_than_points():
    """512 orbitals and 64 points: the products with the orbitals have four column tiles where the plan's others have one."""
    gen = torch.Generator(device=DEV).manual_seed(2)
    phi, psi = (torch.randn(4000, 512, dtype=torch.complex128, device=DEV, generator=gen) for _ in range(2))
    idx = torch.randperm(600, device=DEV, generator=gen)[:64].sort().values
    g = torch.randn(600, 64, dtype=torch.complex128, device=DEV, generator=gen)
    few = _grads(phi[:600].contiguous(), psi[:600].contiguous(), idx, (0, 600), 600, g)
    many = _grads(phi, psi, idx, (0, 600), 4000, g)
    assert torch.equal(few[0], many[0][:600]) and torch.equal(few[1], many[1][:600])
