"""Poisson solves by register lines (complex64, axes up to 64 points) against the oracle: every line length, ragged
column tiles, both tile widths, strided rows, in place.

Tolerance: six line transforms of at most five stages, about 2.5 units of 2^-24 a stage (twiddle and butterfly), relative
to the largest value: 75 2^-24 = 4.5e-6.
"""
import ctypes

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


class _Handle(ctypes.Structure):
    """The head of the library's exchange handle, up to the choice between the three register passes and the five."""
    _fields_ = [("n", ctypes.c_int * 3), ("n_r", ctypes.c_int64), ("cell", ctypes.c_double * 3), ("n_mu", ctypes.c_int),
                ("n_phi", ctypes.c_int), ("n_psi", ctypes.c_int), ("orb_dtype", ctypes.c_int), ("mode", ctypes.c_int),
                ("kind", ctypes.c_int), ("omega", ctypes.c_double), ("q", ctypes.c_double * 3), ("max_rows", ctypes.c_int64),
                ("rd", ctypes.c_int * 39), ("tw", ctypes.c_void_p * 3), ("ktab", ctypes.c_void_p), ("lines", ctypes.c_bool)]


LENGTHS = (8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64)


@pytest.mark.parametrize("axis", [0, 1, 2])
@pytest.mark.parametrize("n", LENGTHS)
def test_register_lines_keep_the_bits_of_the_five_passes(n, axis):
    """complex128 results of the application follow the last bits of V: the register passes round as the passes through
    shared memory do, for every length on every axis."""
    shape = [(9, 8, 10), (10, 9, 8), (8, 10, 9)][n % 3]
    shape = tuple(n if a == axis else s for a, s in enumerate(shape))
    n_mu = 11
    ex = isdf.Exchange(shape, tuple(0.4 * s for s in shape), n_mu, 4, 4, orb_dtype=torch.complex64, mode="mixed",
                       kernel="erfc" if n % 2 else "coulomb", omega=0.25, q=(0.11, 0.0, -0.05))
    h = _Handle.from_address(ex._h.value)
    assert (tuple(h.n), h.n_r, h.n_mu, h.n_phi, h.n_psi, h.mode, h.omega, tuple(h.q)) == (
        shape, int(np.prod(shape)), n_mu, 4, 4, isdf.MIXED, 0.25, (0.11, 0.0, -0.05))
    assert tuple(h.cell) == tuple(0.4 * s for s in shape) and h.tw[0] and h.tw[2] and h.ktab and h.lines
    g = torch.Generator(device=DEV).manual_seed(n)
    theta = torch.randn(h.n_r, n_mu, dtype=torch.complex64, device=DEV, generator=g)
    n0 = isdf.kernel_launches()
    three = ex.potential(theta)
    n1 = isdf.kernel_launches()
    h.lines = False
    five = ex.potential(theta)
    assert (n1 - n0, isdf.kernel_launches() - n1) == (3, 5)
    assert torch.equal(torch.view_as_real(three), torch.view_as_real(five))
