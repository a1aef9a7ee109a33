"""Weights of rows held in registers: bit-equal to the oracle at the edges of the pieces per lane, with zeros, subnormals
and wide ranges inside a row."""
import numpy as np
import pytest
import torch

import oracle as O
import paper_2208_07731_gb300 as isdf

pytestmark = pytest.mark.gpu
DEV = "cuda:0"


def _rows(rng, n_r, n, dtype):
    x = rng.standard_normal((n_r, n)) + 1j * rng.standard_normal((n_r, n))
    tiny = 1e-44 if dtype == np.complex64 else 5e-324
    low = 1e-38 if dtype == np.complex64 else 1e-308
    for r in range(n_r):
        kind = r % 8
        if kind == 1:
            x[r, ::3] = 0.0
        elif kind == 2:
            x[r] *= 2.0 ** rng.integers(-40, 1, n)
        elif kind == 3:
            x[r] *= 2.0 ** rng.integers(-7, 1, n)
        elif kind == 4:
            x[r] = x[r] * low
        elif kind == 5:
            x[r] = tiny * rng.integers(0, 3, n)
        elif kind == 6:
            x[r] = 0.0
    return x.astype(dtype)


@pytest.mark.parametrize("dtype,widths", [
    (np.complex64, (2, 64, 66, 128, 130, 256, 258, 510, 512)),
    (np.complex128, (1, 31, 32, 33, 64, 65, 128, 129, 256)),
])
def test_register_rows_match_oracle(dtype, widths):
    rng = np.random.default_rng(7)
    for n in widths:
        m = max(widths[0], n - 2)
        a, b = _rows(rng, 67, n, dtype), _rows(rng, 67, m, dtype)[::-1].copy()
        A, B = torch.from_numpy(a).to(DEV), torch.from_numpy(b).to(DEV)
        for kind in ("ssm", "psm"):
            assert np.array_equal(isdf.weights(A, B, kind).cpu().numpy(), O.weights(a, b, kind)), (n, kind)
    # a strided view whose rows are aligned, and the running sum of two pairs
    pad = np.zeros((67, 68), dtype)
    pad[:, :60] = _rows(rng, 67, 60, dtype)
    P = torch.from_numpy(pad).to(DEV)[:, :60]
    w = isdf.weights(P, P)
    one = O.weights(pad[:, :60].copy(), pad[:, :60].copy())
    assert np.array_equal(w.cpu().numpy(), one)
    isdf.weights(P, P, out=w, accumulate=True)
    assert np.array_equal(w.cpu().numpy(), one + one)
