"""Poisson solves by register lines (complex64, axes up to 64 points) against the oracle: every line length, ragged
column tiles, both tile widths, strided rows, in place.

Tolerance: six line transforms of at most five stages, about 2.5 units of 2^-24 a stage (twiddle and butterfly), relative
to the largest value: 75 2^-24 = 4.5e-6.
"""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2208_07731_gb300 as isdf

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


@pytest.mark.parametrize("shape,n_mu,kernel,q", [
    ((8, 9, 10), 3, "erfc", None),
    ((12, 15, 16), 33, "coulomb", None),
    ((18, 20, 24), 13, "coulomb", (0.13, -0.07, 0.02)),
    ((25, 27, 30), 9, "erfc", None),
    ((32, 36, 40), 8, "coulomb", None),
    ((45, 48, 48), 5, "erfc", None),      # class of 48 points, 8 columns
    ((50, 54, 60), 5, "coulomb", None),   # class of 64 points, 4 columns
    ((64, 10, 64), 37, "erfc", None),     # class of 64 points, 8 columns
    ((24, 64, 64), 7, "coulomb", None),
])
def test_register_lines_match_oracle(shape, n_mu, kernel, q):
    rng = np.random.default_rng(n_mu)
    n_r, ld = int(np.prod(shape)), n_mu + 2
    cell = tuple(0.4 * s for s in shape)
    buf = (rng.standard_normal((n_r, ld)) + 1j * rng.standard_normal((n_r, ld))).astype(np.complex64)
    ref = O.poisson(buf[:, :n_mu], shape, cell, kernel, 0.3 if kernel == "erfc" else 0.0, q or (0.0, 0.0, 0.0))
    ex = isdf.Exchange(shape, cell, n_mu, 4, 4, orb_dtype=torch.complex64, mode="mixed", kernel=kernel,
                       omega=0.3 if kernel == "erfc" else 0.0, q=q)
    d = torch.from_numpy(buf).to(DEV)
    out = ex.potential(d[:, :n_mu])
    ex.potential(d[:, :n_mu], out=d[:, :n_mu])   # in place, strided
    ex.check()
    assert np.abs(out.cpu().numpy() - ref).max() <= 4.5e-6 * np.abs(ref).max()
    got = d.cpu().numpy()
    assert np.array_equal(got[:, :n_mu], out.cpu().numpy())
    assert np.array_equal(got[:, n_mu:], buf[:, n_mu:])
