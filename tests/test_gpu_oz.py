"""Exact-slicing products: every TMEM accumulation stays an exact integer sum, and row blocks of any size (all group sums
at once, chunks of rows, cut step lists) give the same bits."""
import numpy as np
import pytest
import torch

import paper_2208_07731_gb300 as isdf

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _digits(x, E):
    """The 7 balanced base-256 digits of x relative to 2^E (round half away from zero at 2^(E - 56))."""
    f = [int(abs(v) * 2.0 ** 60 + 0.0) for v in (x * 2.0 ** (-E)).ravel()]   # exact: 53-bit values, |x| < 2^E
    f = [(v + 8) // 16 for v in f]
    f = [v if s >= 0 else -v for v, s in zip(f, x.ravel())]
    d = np.zeros((7, len(f)))
    for i, v in enumerate(f):
        for s in range(6, 0, -1):
            r = ((v + 128) & 255) - 128
            d[s, i] = r
            v = (v - r) >> 8
        d[0, i] = v
    return d.reshape((7,) + x.shape)


def _exact_gram(a):
    """Re and Im of A A^H as the slicing defines it: the pairs s + t <= 8 summed as integers, rounded once."""
    n = a.shape[0]
    E = [int(np.frexp(max(np.abs(r.real).max(), np.abs(r.imag).max()))[1]) for r in a]
    re = np.stack([_digits(r.real, e) for r, e in zip(a, E)], 1)
    im = np.stack([_digits(r.imag, e) for r, e in zip(a, E)], 1)
    out = np.zeros((n, n), dtype=complex)
    S = [[[0] * n for _ in range(n)] for _ in range(2)]
    for g in range(2, 9):
        part = np.zeros((2, n, n))
        for s in range(max(1, g - 7), min(7, g - 1) + 1):
            t = g - s
            part[0] += re[s - 1] @ re[t - 1].T + im[s - 1] @ im[t - 1].T      # exact in FP64: below 2^53
            part[1] += im[s - 1] @ re[t - 1].T - re[s - 1] @ im[t - 1].T
        for p in range(2):
            for i in range(n):
                row = part[p, i]
                Si = S[p][i]
                for j in range(i + 1):
                    Si[j] += int(row[j]) << (8 * (8 - g))
    for i in range(n):
        for j in range(i + 1):
            sc = 2.0 ** (E[i] + E[j] - 64)
            out[i, j] = complex(float(S[0][i][j]) * sc, float(S[1][i][j]) * sc)
    return out


@pytest.mark.parametrize("n_mu,n,kind", [(256, 4096, "same_sign"), (256, 1000, "random"), (300, 272, "same_sign")])
def test_accumulations_are_exact(n_mu, n, kind):
    """Rows whose digits all sit near -128 (leading one near 256) with one sign drive every partial sum to its bound.
    Psi_mu has rows (1, 0, ..., 0), so that M is Phi_mu Phi_mu^H bit for bit."""
    rng = np.random.default_rng(n_mu + n)
    if kind == "same_sign":
        # F = 256 2^48 - 128 (2^40 + ... + 1) + a little: d_1 = 256 or 255, the others in {-128, .., -125}
        base = (256 << 48) - 128 * sum(1 << (8 * k) for k in range(6))
        f = base - (rng.integers(0, 2, (n_mu, n, 2)).astype(np.int64) << 48)
        for k in range(1, 6):   # digit 7 stays: 53-bit mantissas keep the top 53 of 56 bits
            f = f + (rng.integers(0, 4, (n_mu, n, 2)).astype(np.int64) << (8 * k))
        x = (f & ~np.int64(7)).astype(np.float64) * 2.0 ** -56
        a = x[..., 0] + 1j * x[..., 1]
    else:
        a = rng.standard_normal((n_mu, n)) + 1j * rng.standard_normal((n_mu, n))
    psi = np.zeros((n_mu, n), dtype=complex)
    psi[:, 0] = 1.0
    idx = torch.arange(n_mu, device=DEV)
    plan = isdf.Plan(torch.from_numpy(a).to(DEV), torch.from_numpy(psi).to(DEV), idx, mode="fp64")
    M = plan.matrix("M").cpu().numpy()
    low = np.tril_indices(n_mu, -1)
    ref = _exact_gram(a)
    assert np.array_equal(M[low], ref[low])
    assert np.array_equal(np.diag(M).real, np.diag(ref).real)


@pytest.mark.parametrize("n_r,n,n_mu", [(3000, 17, 129), (2500, 40, 300), (60000, 20, 130)])
def test_row_blocks_agree(n_r, n, n_mu):
    """Small row blocks and one block over all rows: identical Theta."""
    g = torch.Generator(device=DEV).manual_seed(n)
    phi, psi = (torch.randn(n_r, n, dtype=torch.complex128, device=DEV, generator=g) for _ in range(2))
    idx = torch.randperm(n_r, device=DEV, generator=g)[:n_mu].sort().values
    small = isdf.Plan(phi, psi, idx, mode="fp64", max_rows=200)
    large = isdf.Plan(phi, psi, idx, mode="fp64", max_rows=n_r)
    a, b = small.fit_theta(), large.fit_theta()
    small.check(), large.check()
    assert torch.equal(torch.view_as_real(a), torch.view_as_real(b))
