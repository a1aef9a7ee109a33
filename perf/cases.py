"""What this framework is timed on: calls that its users make, over the sizes they make them at.

A case is a dict of plain values. listed() gives the fixed cases, draw(rng) one more of the same ranges,
prepare(case, seed) what a program holds before the call (orbitals, interpolation points, a plan), run(state) one
pass through the package's entry points with its outputs, work(case) the bytes and operations the pass cannot do
without, exact(case, seed) the same outputs from plain torch in 64 bits.

Inputs: plane-wave Bloch orbitals like those of workload.py (damped random coefficients inside a cutoff sphere, times
a Bloch phase), generated on the GPU and normalised one by one. Points: a shifted low-discrepancy sequence over the
cell, as evenly spread as K-means leaves them.
"""
from __future__ import annotations

import math

import numpy as np
import torch

import paper_2208_07731_gb300 as isdf

DEV = "cuda"
SPACING = 0.375   # grid spacing in bohr (48 points over 18 bohr)


def listed():
    return [
        # a whole decomposition of a tiny cell in FP64, plan and all: the smallest call, latency and launches
        {"name": "decompose_tiny_fp64", "kind": "decompose", "nx": 24, "ny": 24, "nz": 24, "n": 16, "n_mu": 128,
         "iters": 50, "dtype": "c128", "mode": "fp64"},
        # one step of an MD or SCF loop on a medium cell: weight, K-means, new points in a kept plan, Theta
        {"name": "md_step_medium", "kind": "step", "nx": 48, "ny": 48, "nz": 48, "n": 128, "n_mu": 1024,
         "iters": 100, "dtype": "c128", "mode": "mixed"},
        # the K-means weight of a water-box-sized orbital pair: one pass over the orbitals
        {"name": "weights_waterbox", "kind": "weights", "nx": 96, "ny": 96, "nz": 96, "n": 256, "dtype": "c64",
         "weight": "ssm", "alpha": 2.0},
        # the interpolation points of the largest cell
        {"name": "kmeans_silica", "kind": "kmeans", "nx": 128, "ny": 128, "nz": 128, "n_mu": 4096, "iters": 100,
         "early_stop": False},
        # new interpolation points in a kept plan at the largest n_mu: M, its Cholesky factor and inverse in FP64,
        # and the tensor-core operands
        {"name": "update_large", "kind": "update", "nx": 64, "ny": 64, "nz": 64, "n": 1024, "n_mu": 4096,
         "dtype": "c64", "mode": "mixed"},
        # Theta of one default row block of a plan at the largest sizes: the two big tensor-core products
        {"name": "fit_large_mixed", "kind": "fit", "nx": 64, "ny": 64, "nz": 64, "n": 1024, "n_mu": 4096,
         "row_begin": 131072, "rows": 65536, "dtype": "c64", "mode": "mixed"},
        # Theta rows of a water box on a ragged window
        {"name": "fit_waterbox_mixed", "kind": "fit", "nx": 96, "ny": 96, "nz": 96, "n": 256, "n_mu": 2048,
         "row_begin": 400001, "rows": 200003, "dtype": "c64", "mode": "mixed"},
        # Theta in FP64, for programs that need the last digits; sizes that fill no tile
        {"name": "fit_fp64", "kind": "fit", "nx": 45, "ny": 48, "nz": 50, "n": 120, "n_mu": 1000,
         "row_begin": 0, "rows": 108000, "dtype": "c128", "mode": "fp64"},
        # loss and orbital gradients of the exchange-like surrogate, tensor-core adjoint
        {"name": "grad_mixed", "kind": "grad", "nx": 48, "ny": 48, "nz": 48, "n": 192, "n_mu": 1536,
         "dtype": "c64", "mode": "mixed"},
        # Theta inside torch.autograd in FP64: forward and backward of a small problem
        {"name": "autograd_fp64", "kind": "autograd", "nx": 32, "ny": 32, "nz": 32, "n": 48, "n_mu": 320,
         "dtype": "c128", "mode": "fp64"},
        # the exchange operator with the fitted vectors: Poisson solves by FFT, then the application
        {"name": "exchange_medium", "kind": "exchange", "nx": 48, "ny": 48, "nz": 48, "n": 128, "n_mu": 1024,
         "dtype": "c64", "mode": "mixed", "kernel": "erfc", "omega": 0.106},
        # eight k-points of one cell at shared points: many small problems side by side
        {"name": "batch_kpoints", "kind": "batch", "nx": 48, "ny": 48, "nz": 48, "n": 32, "n_mu": 256, "count": 8,
         "dtype": "c128", "mode": "mixed"},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _grid(rng, lo, hi):
    """Three axis lengths around a common edge, odd ones among them."""
    edge = _log_int(rng, lo, hi)
    return tuple(min(hi, max(lo, edge + rng.choice([0, 0, 1, -1, 2, 3, -3, 4]))) for _ in range(3))


def _cost(case):
    """Rough time in arbitrary units (ms), to keep drawn cases below the largest listed one."""
    w = work(case)
    ms = w["bytes"] / 2.0e9
    if case["kind"] == "kmeans":
        return ms + 2.0e-7 * case["iters"] * case["nx"] * case["ny"] * case["nz"]
    grad = case["kind"] in ("grad", "autograd")
    rate = (2.2e11 if grad else 5.0e11) if case.get("mode") == "mixed" else (1.9e9 if grad else 1.6e10)   # per ms
    extra = 0.0
    if case["kind"] in ("decompose", "step", "update", "autograd", "batch"):
        extra = 5.5 * (case["n_mu"] / 1024.0) ** 1.55 * case.get("count", 1)
    return ms + w["flops"] / rate + extra


def draw(rng):
    """One more case of the listed ranges (24^3 to 128^3 points, 16 to 1024 orbitals, 64 to 4096 points)."""
    cap = max(_cost(c) for c in listed())
    while True:
        kind = rng.choice(["decompose", "step", "weights", "kmeans", "update", "fit", "fit", "grad", "autograd",
                           "exchange", "batch"])
        case = {"kind": kind}
        if kind == "kmeans":
            nx, ny, nz = _grid(rng, 24, 128)
            n_r = nx * ny * nz
            case.update(nx=nx, ny=ny, nz=nz, n_mu=_log_int(rng, 64, min(4096, n_r // 64)),
                        iters=rng.choice([20, 50, 100]), early_stop=rng.random() < 0.5)
        elif kind == "weights":
            nx, ny, nz = _grid(rng, 24, 96)
            case.update(nx=nx, ny=ny, nz=nz, n=_log_int(rng, 16, 512), dtype=rng.choice(["c128", "c64"]))
            case.update(weight=rng.choice(["ssm", "ssm", "ssm", "psm"]), alpha=2.0)
            if case["weight"] == "ssm" and rng.random() < 0.25:
                case["alpha"] = rng.choice([1.0, 3.0, 4.0])
        else:
            hi = {"decompose": 40, "step": 64, "update": 64, "fit": 96, "grad": 56, "autograd": 40, "exchange": 64,
                  "batch": 48}[kind]
            nx, ny, nz = _grid(rng, 24, hi)
            n_r = nx * ny * nz
            mode = "fp64" if kind == "autograd" else rng.choice(["mixed", "mixed", "fp64"])
            n_hi = {"decompose": 64, "batch": 64, "autograd": 64, "exchange": 256, "grad": 256}.get(kind, 1024)
            n = _log_int(rng, 16, n_hi)
            if mode == "mixed":
                n = max(32, n // 32 * 32)
            n_mu = min(4096, n_r // 64, n * n // 2, int(n * rng.uniform(3.0, 9.0)))
            if mode == "mixed":
                n_mu = n_mu // 64 * 64
            if n_mu < 64:
                continue
            case.update(nx=nx, ny=ny, nz=nz, n=n, n_mu=n_mu, dtype=rng.choice(["c128", "c64"]), mode=mode)
            if kind in ("decompose", "step"):
                case["iters"] = rng.choice([20, 50, 100])
            elif kind == "fit":
                rows = min(n_r, _log_int(rng, 1000, 262144))
                case.update(rows=rows, row_begin=rng.randint(0, n_r - rows))
            elif kind == "exchange":
                # axes of the FFT are products of 2, 3 and 5
                fft = [24, 25, 27, 30, 32, 36, 40, 45, 48, 50, 54, 60, 64]
                nx, ny, nz = (min(fft, key=lambda f: abs(f - m)) for m in (nx, ny, nz))
                n_mu = min(n_mu, nx * ny * nz // 64)
                case.update(nx=nx, ny=ny, nz=nz, n_mu=n_mu // 64 * 64 if mode == "mixed" else n_mu)
                case.update(kernel=rng.choice(["erfc", "coulomb"]), omega=0.106)
            elif kind == "batch":
                case["count"] = rng.randint(2, 8)
        if _memory(case) <= 40e9 and _cost(case) <= cap:
            return case


def _memory(case):
    """Rough bytes of a prepared case and its outputs."""
    n_r, n, m = case["nx"] * case["ny"] * case["nz"], case.get("n", 0), case.get("n_mu", 0)
    if case["kind"] in ("kmeans", "weights"):
        return n_r * (64 + 32 * n)
    c = case.get("count", 1)
    return c * (n_r * n * 64.0 + 12 * 16.0 * m * m + 16.0 * min(n_r, 65536) * m * 8 + 16.0 * n_r * m * 2)


# ---------------------------------------------------------------- inputs

def _shape(case):
    return case["nx"], case["ny"], case["nz"]


def _cell(case):
    return tuple(SPACING * n for n in _shape(case))


def _orbitals(case, gen, k=(0.25, 0.25, 0.0)):
    """n_r x n orbitals: damped random plane waves in a sphere of 0.75 of the grid's band limit, Bloch phase k (in
    units of 2 pi / L), each of norm 1 over the cell."""
    nx, ny, nz = _shape(case)
    n, cd = case["n"], torch.complex128 if case["dtype"] == "c128" else torch.complex64
    rd = torch.float64 if cd == torch.complex128 else torch.float32
    freq = [torch.fft.fftfreq(m, 1.0 / m, device=DEV, dtype=torch.float64) * (2.0 * math.pi / (SPACING * m))
            for m in (nx, ny, nz)]
    g2 = freq[0][:, None, None] ** 2 + freq[1][None, :, None] ** 2 + freq[2][None, None, :] ** 2
    damp = torch.where(g2 <= (0.75 * math.pi / SPACING) ** 2, torch.exp(-g2 / 4.0), torch.zeros_like(g2)).to(rd)
    ph = [torch.exp(2j * math.pi * kf / m * torch.arange(m, device=DEV, dtype=torch.float64))
          for kf, m in zip(k, (nx, ny, nz))]
    phase = (ph[0][:, None, None] * ph[1][None, :, None] * ph[2][None, None, :]).to(cd)
    out = torch.empty((nx * ny * nz, n), dtype=cd, device=DEV)
    for a in range(0, n, 64):
        b = min(n, a + 64)
        c = torch.randn((b - a, nx, ny, nz, 2), generator=gen, device=DEV, dtype=rd)
        f = torch.fft.fftn(torch.view_as_complex(c) * damp, dim=(1, 2, 3)) * phase
        f = f.reshape(b - a, -1)
        f /= torch.linalg.vector_norm(f, dim=1, keepdim=True) * SPACING ** 1.5
        out[:, a:b] = f.T
    return out


def _pair(case, gen, k=(0.25, 0.25, 0.0)):
    return _orbitals(case, gen, k), _orbitals(case, gen, k)


def _points(case, seed, n_mu=None):
    """n_mu distinct grid indices spread over the cell: the additive sequence of the 3-D golden ratio, shifted."""
    nx, ny, nz = _shape(case)
    m = n_mu or case["n_mu"]
    g = 1.2207440846057596
    shift = np.random.default_rng(seed).random(3)
    t = np.arange(4 * m + 64)[:, None] * np.array([1 / g, 1 / g ** 2, 1 / g ** 3])[None, :] + shift
    ijk = np.floor((t % 1.0) * np.array([nx, ny, nz])).astype(np.int64)
    flat = (ijk[:, 0] * ny + ijk[:, 1]) * nz + ijk[:, 2]
    _, first = np.unique(flat, return_index=True)
    return torch.from_numpy(np.sort(flat[np.sort(first)[:m]])).to(DEV)


def _density(case, gen):
    """A smooth positive weight: Gaussian atoms on a 6 x 6 x 6 lattice over the density of a few random waves."""
    nx, ny, nz = _shape(case)
    small = dict(case, n=8, dtype="c64")
    w = _orbitals(small, gen).abs().square().sum(1).double().reshape(nx, ny, nz)
    w *= 8.0 / w.mean()
    for axis, m in enumerate((nx, ny, nz)):
        u = torch.arange(m, device=DEV, dtype=torch.float64) / m
        d = ((u[:, None] - (torch.arange(6, device=DEV) + 0.5) / 6 + 0.5) % 1.0 - 0.5) * SPACING * m
        f = torch.exp(-0.5 * d * d).sum(1)
        g = f if axis == 0 else g[..., None] * f
    return (w + 60.0 * g).reshape(-1).contiguous()


def _start_points(w, n_mu, gen):
    """Weighted-random distinct start points (smallest -ln(u) / w)."""
    u = 1.0 - torch.rand(w.numel(), generator=gen, device=DEV, dtype=torch.float64)
    return torch.sort(torch.topk(-torch.log(u) / w, n_mu, largest=False).indices).values


def _loss_matrix(n_mu, gen):
    """Hermitian positive matrix of the surrogate loss."""
    a = torch.randn((n_mu, n_mu, 2), generator=gen, device=DEV, dtype=torch.float64)
    a = torch.view_as_complex(a) / math.sqrt(2.0 * n_mu)
    return (a + a.conj().T + 5.0 * torch.eye(n_mu, device=DEV)).contiguous()


def _inputs(case, seed):
    gen = torch.Generator(device=DEV).manual_seed(seed)
    kind, s = case["kind"], {}
    if kind == "kmeans":
        s["w"] = _density(case, gen)
        s["init"] = _start_points(s["w"], case["n_mu"], gen)
        return s
    if kind == "batch":
        s["pairs"] = [_pair(case, gen, (0.125 * (b % 4), 0.125 * (b // 4), 0.0)) for b in range(case["count"])]
        s["idx"] = _points(case, seed)
        return s
    s["phi"], s["psi"] = _pair(case, gen)
    if kind in ("decompose", "step"):
        w = s["phi"].abs().square().sum(1) + s["psi"].abs().square().sum(1)
        s["init"] = _start_points(w.double(), case["n_mu"], gen)
    elif kind != "weights":
        s["idx"] = _points(case, seed)
    if kind == "grad":
        s["K"] = _loss_matrix(case["n_mu"], gen)
    elif kind in ("autograd", "exchange"):
        cd = torch.complex64 if case["mode"] == "mixed" else torch.complex128
        rd = torch.float32 if cd == torch.complex64 else torch.float64
        shape = (s["phi"].shape[0], case["n_mu"], 2)
        s["theta" if kind == "exchange" else "grad"] = torch.view_as_complex(
            torch.randn(shape, generator=gen, device=DEV, dtype=rd))
    return s


def prepare(case, seed):
    s = _inputs(case, seed)
    s["case"] = case
    kind = case["kind"]
    if kind == "step":
        s["plan"] = isdf.Plan(s["phi"], s["psi"], _points(case, seed), mode=case["mode"])
    elif kind in ("update", "fit", "grad"):
        s["plan"] = isdf.Plan(s["phi"], s["psi"], s["idx"], mode=case["mode"])
        if kind == "update":
            s["idx"] = _points(case, seed + 1)   # the points of the next step
    elif kind == "exchange":
        s["ex"] = isdf.Exchange(_shape(case), _cell(case), case["n_mu"], case["n"], case["n"],
                                orb_dtype=s["phi"].dtype, mode=case["mode"], kernel=case["kernel"],
                                omega=case["omega"])
    elif kind == "batch":
        s["batch"] = isdf.Batch(s["pairs"], s["idx"], mode=case["mode"])
        s["idx"] = _points(case, seed + 1)
    return s


# ---------------------------------------------------------------- one pass

def run(s):
    c = s["case"]
    kind = c["kind"]
    if kind == "decompose":
        r = isdf.decompose(s["phi"], s["psi"], _shape(c), _cell(c), c["n_mu"], s["init"], c["iters"], mode=c["mode"])
        return dict(r["kmeans"], w=r["w"], theta=r["theta"])
    if kind == "step":
        w = isdf.weights(s["phi"], s["psi"])
        km = isdf.kmeans(w, _shape(c), _cell(c), c["n_mu"], s["init"], c["iters"])
        s["plan"].update(km["idx"])
        return dict(km, w=w, theta=s["plan"].fit_theta())
    if kind == "weights":
        return isdf.weights(s["phi"], s["psi"], c["weight"], c["alpha"])
    if kind == "kmeans":
        return isdf.kmeans(s["w"], _shape(c), _cell(c), c["n_mu"], s["init"], c["iters"],
                           early_stop=c["early_stop"])
    if kind == "update":
        s["plan"].update(s["idx"])
        return {m: s["plan"].matrix(m) for m in ("M", "L", "Minv")}
    if kind == "fit":
        return s["plan"].fit_theta(c["row_begin"], c["rows"])
    if kind == "grad":
        loss, gphi, gpsi = isdf.surrogate_loss_and_grad(s["plan"], s["K"], SPACING ** 3)
        return {"loss": loss, "grad_phi": gphi, "grad_psi": gpsi}
    if kind == "autograd":
        phi, psi = s["phi"].detach().requires_grad_(), s["psi"].detach().requires_grad_()
        theta = isdf.ISDFThetaFn.apply(phi, psi, s["idx"], c["mode"])
        gphi, gpsi = torch.autograd.grad(theta, (phi, psi), s["grad"])
        return {"theta": theta.detach(), "grad_phi": gphi, "grad_psi": gpsi}
    if kind == "exchange":
        v = s["ex"].potential(s["theta"])
        return {"v": v, "vx": s["ex"].apply(s["phi"], s["psi"], s["idx"], v)}
    if kind == "batch":
        s["batch"].update(s["idx"])
        return s["batch"].fit_theta()
    raise ValueError(kind)


# ---------------------------------------------------------------- what a pass cannot do without

def work(case):
    kind = case["kind"]
    n_r = case["nx"] * case["ny"] * case["nz"]
    n, m = float(case.get("n", 0)), float(case.get("n_mu", 0))
    eo = 16 if case.get("dtype") == "c128" else 8          # orbital entry
    et = 8 if case.get("mode") == "mixed" else 16          # Theta entry
    orb = 2.0 * n_r * n * eo                               # both orbital sets
    chol = 4.0 * m ** 3                                    # factor, triangular inverse, L^-H L^-1 (complex)
    fit_row = 16.0 * n * m + 8.0 * m * m                   # two Gram products and Y M^-1, per grid row
    m_flops = 16.0 * n * m * m / 2                         # M: lower triangle of two Gram products
    km = {"bytes": n_r * 8.0 + m * 8 + m * 32 + n_r * 4.0, "flops": 8.0 * n_r * case.get("iters", 0)}
    if kind == "weights":
        return {"bytes": orb + 8.0 * n_r, "flops": 4.0 * 2 * n_r * n}
    if kind == "kmeans":
        # every point is looked at in every pass; the nearest centroids are a few of n_mu
        return km
    if kind in ("decompose", "step"):
        return {"bytes": orb + 12.0 * n_r + n_r * m * et,
                "flops": 8.0 * n_r * n + km["flops"] + m_flops + chol + n_r * fit_row}
    if kind == "update":
        return {"bytes": orb + 3 * m * m * 16 + m * 8, "flops": m_flops + chol}
    if kind == "fit":
        rows = case["rows"]
        return {"bytes": 2.0 * rows * n * eo + 2 * m * n * 16 + m * m * 16 + rows * m * et, "flops": rows * fit_row}
    if kind in ("grad", "autograd"):
        # P^phi, P^psi, Theta, (G,) Ybar, Mbar and the four products with the orbitals
        g = 8.0 * m * m * (4 if kind == "grad" else 3) + 48.0 * n * m
        io = orb + 2.0 * n_r * n * 16 + (m * m * 16 if kind == "grad" else n_r * m * et * 2.0)
        extra = m_flops + chol if kind == "autograd" else 0.0
        return {"bytes": io, "flops": n_r * g + extra}
    if kind == "exchange":
        fft = 2 * 5.0 * n_r * math.log2(n_r) * m
        return {"bytes": 2.0 * n_r * m * et + orb + n_r * n * 16, "flops": fft + 16.0 * n_r * n * m}
    if kind == "batch":
        return {"bytes": case["count"] * (orb + n_r * m * et),
                "flops": case["count"] * (m_flops + chol + n_r * fit_row)}
    raise ValueError(kind)


# ---------------------------------------------------------------- 64-bit values

def _theta64(phi, psi, idx, rows=slice(None)):
    """Theta = Y M^-1 of some rows, with Y = (Phi Phi_mu^H) o conj(Psi Psi_mu^H) and M its rows at idx."""
    pm, qm = phi[idx].to(torch.complex128), psi[idx].to(torch.complex128)
    M = (pm @ pm.conj().T) * (qm @ qm.conj().T).conj()
    out = []
    minv = torch.linalg.inv(M)
    minv = 0.5 * (minv + minv.conj().T)
    P, Q = phi[rows], psi[rows]
    for a in range(0, P.shape[0], 32768):
        p, q = P[a:a + 32768].to(torch.complex128), Q[a:a + 32768].to(torch.complex128)
        out.append(((p @ pm.conj().T) * (q @ qm.conj().T).conj()) @ minv)
    return torch.cat(out)


def _weights64(c, phi, psi):
    def moment(x):
        x = x.to(torch.complex128)
        s = x.real.square() + x.imag.square()
        a = c.get("alpha", 2.0)
        return (s if a == 2.0 else s ** (a / 2.0)).sum(1)
    p, q = moment(phi), moment(psi)
    return p * q if c.get("weight") == "psm" else p + q


def _gradients64(s, plan_grad=None):
    """Orbital gradients by torch autograd through the formulas of Theta, in row blocks."""
    idx = s["idx"]
    phi, psi = s["phi"].to(torch.complex128), s["psi"].to(torch.complex128)
    pm, qm = phi[idx].requires_grad_(), psi[idx].requires_grad_()
    loss, gp, gq = 0.0, torch.zeros_like(phi), torch.zeros_like(psi)
    M = (pm @ pm.conj().T) * (qm @ qm.conj().T).conj()
    W = torch.linalg.inv(M)
    Wl = W.detach().requires_grad_()
    pl, ql = pm.detach().requires_grad_(), qm.detach().requires_grad_()
    theta = []
    for a in range(0, phi.shape[0], 16384):
        p = phi[a:a + 16384].clone().requires_grad_()
        q = psi[a:a + 16384].clone().requires_grad_()
        th = ((p @ pl.conj().T) * (q @ ql.conj().T).conj()) @ Wl
        if plan_grad is None:
            part = SPACING ** 3 * (th.conj() * (th @ s["K"].T)).real.sum()
            part.backward()
            loss = loss + part.detach()
        else:
            th.backward(plan_grad[a:a + 16384].to(torch.complex128))
            theta.append(th.detach())
        gp[a:a + 16384], gq[a:a + 16384] = p.grad, q.grad
    gm = torch.autograd.grad(W, (pm, qm), Wl.grad)
    gp.index_add_(0, idx, gm[0] + pl.grad)
    gq.index_add_(0, idx, gm[1] + ql.grad)
    return loss, gp, gq, theta


def exact(case, seed):
    kind = case["kind"]
    s = None if kind == "kmeans" else _inputs(case, seed)
    if kind == "weights":
        return _weights64(case, s["phi"], s["psi"])
    if kind == "kmeans":
        return None   # whole numbers, and centroids that follow from exact integer sums
    if kind in ("decompose", "step"):
        # the points are whole numbers that the rest hangs on; the weight has a value of its own
        out = {k: None for k in ("idx", "centroids", "objective", "labels", "stats")}
        return dict(out, w=_weights64({}, s["phi"], s["psi"]), theta=None)
    if kind == "update":
        idx = _points(case, seed + 1)
        pm, qm = s["phi"][idx].to(torch.complex128), s["psi"][idx].to(torch.complex128)
        M = (pm @ pm.conj().T) * (qm @ qm.conj().T).conj()
        return {"M": M, "L": torch.linalg.cholesky(M), "Minv": torch.linalg.inv(M)}
    if kind == "fit":
        if work(case)["flops"] > 1.5e13:   # over 20 seconds on the FP64 pipe
            return None
        a = case["row_begin"]
        return _theta64(s["phi"], s["psi"], s["idx"], slice(a, a + case["rows"]))
    if kind == "grad":
        loss, gp, gq, _ = _gradients64(s)
        return {"loss": loss.reshape(1), "grad_phi": gp, "grad_psi": gq}
    if kind == "autograd":
        _, gp, gq, theta = _gradients64(s, s["grad"])
        return {"theta": torch.cat(theta), "grad_phi": gp, "grad_psi": gq}
    if kind == "exchange":
        shape, cell = _shape(case), _cell(case)
        freq = [torch.fft.fftfreq(m, 1.0 / m, device=DEV, dtype=torch.float64) * (2 * math.pi / L)
                for m, L in zip(shape, cell)]
        g2 = freq[0][:, None, None] ** 2 + freq[1][None, :, None] ** 2 + freq[2][None, None, :] ** 2
        zero = g2 == 0
        g2s = torch.where(zero, torch.ones_like(g2), g2)
        if case["kernel"] == "erfc":
            om = case["omega"]
            k = torch.where(zero, torch.full_like(g2, math.pi / om ** 2),
                            -4 * math.pi * torch.expm1(-g2s / (4 * om * om)) / g2s)
        else:
            k = torch.where(zero, torch.zeros_like(g2), 4 * math.pi / g2s)
        v = torch.empty(s["theta"].shape, dtype=torch.complex128, device=DEV)
        for a in range(0, case["n_mu"], 64):
            t = s["theta"][:, a:a + 64].T.to(torch.complex128).reshape((-1,) + shape)
            t = torch.fft.ifftn(torch.fft.fftn(t, dim=(1, 2, 3)) * k, dim=(1, 2, 3))
            v[:, a:a + 64] = t.reshape(t.shape[0], -1).T
        pm, qm = s["phi"][s["idx"]].to(torch.complex128), s["psi"][s["idx"]].to(torch.complex128)
        vx = torch.empty((v.shape[0], case["n"]), dtype=torch.complex128, device=DEV)
        for a in range(0, v.shape[0], 32768):
            p = s["phi"][a:a + 32768].to(torch.complex128)
            vx[a:a + 32768] = -((v[a:a + 32768] * (p @ pm.conj().T)) @ qm)
        return {"v": v, "vx": vx}
    if kind == "batch":
        idx = _points(case, seed + 1)
        return [_theta64(p, q, idx) for p, q in s["pairs"]]
    raise ValueError(kind)
