"""The last bits of a plan's M, L and M^-1. In ISDF_MIXED mode the FP16 digits of M^-1 follow them, and the complex128
gradients of that mode follow the digits (one digit that falls the other way moves entries by up to 1e-7), so the order in
which these matrices' terms are added is held to recorded values: tests/golden/plan_bits.json has the SHA-256 of each
matrix's bytes for orbitals made of integer arithmetic alone. Sizes: one tile and ragged ones, general and exact-slicing
products, split sums in the triangular inverse (128 rows), the recursive factorisation with ragged halves."""
import hashlib
import json
import os

import numpy as np
import pytest
import torch

import paper_2208_07731_gb300 as isdf

pytestmark = pytest.mark.gpu
GOLDEN = os.path.join(os.path.dirname(os.path.abspath(__file__)), "golden", "plan_bits.json")
CASES = [("fp64", 12, 37, "tensor"), ("fp64", 24, 200, "tensor"), ("fp64", 40, 333, "simt"), ("mixed", 32, 64, "tensor"),
         ("mixed", 64, 256, "tensor"), ("mixed", 64, 512, "tensor"), ("mixed", 64, 640, "simt"), ("mixed", 96, 832, "tensor"),
         ("mixed", 128, 1088, "tensor"), ("mixed", 192, 1536, "tensor")]


def orbitals(seed, rows, n):
    """rows x n complex128, both parts multiples of 2^-52 in [-1, 1): the splitmix64 sequence."""
    with np.errstate(over="ignore"):
        z = (np.arange(1, 2 * rows * n + 1, dtype=np.uint64) + np.uint64(seed << 32)) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z ^= z >> np.uint64(31)
    x = (z >> np.uint64(11)).astype(np.float64) * 2.0 ** -52 - 1.0
    return torch.from_numpy(x.view(np.complex128).reshape(rows, n))


def digests(mode, n, n_mu, products):
    phi, psi = (orbitals(s, n_mu + 5, n).cuda() for s in (n_mu, n_mu + 1))
    plan = isdf.Plan(phi, psi, torch.arange(n_mu + 4, 4, -1), mode=mode, fp64_products=products)
    plan.check()
    return {m: hashlib.sha256(plan.matrix(m).cpu().numpy().tobytes()).hexdigest() for m in ("M", "L", "Minv")}


@pytest.mark.parametrize("case", CASES, ids=lambda c: "-".join(map(str, c)))
def test_matrices_keep_their_bits(case):
    with open(GOLDEN) as f:
        assert digests(*case) == json.load(f)["-".join(map(str, case))]
