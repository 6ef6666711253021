"""Performance cases of the HOTRG library: what its users have it compute.

A solve is a chain of half-steps, and a half-step is an environment, an
isometry and a contraction, all of them made of matrix products.  The cases
time those parts through the component calls of ``Solver`` on tensors that
stay on the device, and two whole solves.  Sizes are those of the repository's
own workloads (Ising Dcut 16 to 64, the odd bond dimensions that multiplet
cuts leave in XY and Potts runs), in FP64, which is the default precision, and
in split precision with 3 to 5 slices (4 is the default).

Inputs have the shape of the method's own: site tensors whose entries fall off
with every leg index and vanish where the parities of the legs do not add up
(the Z2 rule of the Ising tensor), isometries that are concentrated on the
low index pairs, environments with an algebraically falling spectrum.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2306_00358_gb300 import Solver

DEVICE = "cuda"
BETA_C = 0.5 * math.log(1.0 + math.sqrt(2.0))


def listed():
    return [
        # one small product in the default precision: a call's fixed cost
        {"name": "gemm_fp64_96x80x72", "kind": "gemm", "precision": "fp64", "slices": 4, "m": 96, "n": 80, "k": 72},
        # the product bench.py calibrates the split path with
        {"name": "gemm_split_16384x4096x4096", "kind": "gemm", "precision": "split", "slices": 4, "m": 16384,
         "n": 4096, "k": 4096},
        # environment of a mid-flow tensor with unequal legs, Dcut 24 of the serving mix
        {"name": "env_fp64_24x22", "kind": "environment", "precision": "fp64", "slices": 4, "dx": 24, "dy": 22},
        # environment of the headline half-step (Ising, Dcut 64)
        {"name": "env_split_64", "kind": "environment", "precision": "split", "slices": 4, "dx": 64, "dy": 64},
        # isometry of the smallest configuration (Ising, Dcut 16, FP64)
        {"name": "iso_fp64_n256_d16", "kind": "isometry", "precision": "fp64", "slices": 4, "n": 256, "dcut": 16},
        # isometry of the coupling sweep's Dcut 32
        {"name": "iso_split_n1024_d32", "kind": "isometry", "precision": "split", "slices": 4, "n": 1024, "dcut": 32},
        # isometry of the headline half-step
        {"name": "iso_split_n4096_d64", "kind": "isometry", "precision": "split", "slices": 4, "n": 4096, "dcut": 64},
        # contraction of an FP64 reference half-step at Dcut 48
        {"name": "contract_fp64_48", "kind": "contract", "precision": "fp64", "slices": 4, "dx": 48, "dy": 48,
         "dn": 48},
        # contraction with the odd bond dimensions of a multiplet cut (XY, Dcut 48)
        {"name": "contract_split_45x43_47", "kind": "contract", "precision": "split", "slices": 4, "dx": 45, "dy": 43,
         "dn": 47},
        # contraction of the headline half-step, the largest call
        {"name": "contract_split_64", "kind": "contract", "precision": "split", "slices": 4, "dx": 64, "dy": 64,
         "dn": 64},
        # the smallest configuration, whole: 40 half-steps to a 2^20 x 2^20 lattice
        {"name": "solve_fp64_d16", "kind": "solve", "precision": "fp64", "slices": 4, "beta": 0.44, "h": 0.0,
         "dcut": 16, "nsteps": 40},
        # one run of the coupling sweep, whole
        {"name": "solve_split_d32", "kind": "solve", "precision": "split", "slices": 4, "beta": BETA_C, "h": 1e-3,
         "dcut": 32, "nsteps": 40},
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(("gemm", "environment", "isometry", "contract", "contract", "solve"))
    precision = rng.choice(("fp64", "split"))
    case = {"kind": kind, "precision": precision, "slices": rng.choice((3, 4, 4, 4, 5)) if precision == "split" else 4}
    split = precision == "split"
    if kind == "gemm":
        # FP64 products stay below the FP64 contraction's cost
        while True:
            m, n, k = (_log_int(rng, 1, 16384 if split else 4096), _log_int(rng, 1, 4096),
                       _log_int(rng, 1, 4096))
            if m * n * k >= 64:
                return {**case, "m": m, "n": n, "k": k}
    if kind == "environment":
        top = 64 if split else 40
        return {**case, "dx": _log_int(rng, 6, top), "dy": _log_int(rng, 6, top)}
    if kind == "isometry":
        dx = _log_int(rng, 8, 64 if split else 40)
        return {**case, "n": dx * dx, "dcut": rng.randint(max(4, dx // 2), min(64, dx))}
    if kind == "contract":
        top = 64 if split else 44
        dx, dy = _log_int(rng, 6, top), _log_int(rng, 6, top)
        return {**case, "dx": dx, "dy": dy, "dn": min(dx * dx, _log_int(rng, max(4, dx // 2), top))}
    return {**case, "beta": round(rng.uniform(0.40, 0.48), 4), "h": rng.choice((0.0, 1e-3)),
            "dcut": rng.randint(8, 32 if split else 24), "nsteps": rng.randint(20, 40)}


# ------------------------------------------------------------------ inputs
def _generator(seed):
    return torch.Generator(device=DEVICE).manual_seed(int(seed))


def _normal(shape, gen):
    return torch.randn(shape, generator=gen, device=DEVICE, dtype=torch.float64)


def _fall(n, power):
    return (1.0 + torch.arange(n, device=DEVICE, dtype=torch.float64)) ** -power


def _site_tensor(dx, dy, seed):
    """(dx, dy, dx, dy): entries fall off with each leg, odd total parity is zero, largest entry 1."""
    t = _normal((dx, dy, dx, dy), _generator(seed))
    for leg, n in enumerate(t.shape):
        shape = [1, 1, 1, 1]
        shape[leg] = n
        t *= _fall(n, 0.75).reshape(shape)
    px = (torch.arange(dx, device=DEVICE) % 2).to(torch.int64)
    py = (torch.arange(dy, device=DEVICE) % 2).to(torch.int64)
    odd = (px[:, None, None, None] + py[None, :, None, None] + px[None, None, :, None] + py) % 2
    t = torch.where(odd == 0, t, torch.zeros_like(t))
    return (t / t.abs().max()).contiguous()


def _isometry(dx, dn, seed):
    """(dx, dx, dn), orthonormal columns concentrated on the low index pairs."""
    w = _fall(dx, 0.75)
    g = _normal((dx * dx, dn), _generator(seed + 7919)) * (w[:, None] * w).reshape(-1, 1)
    q, _ = torch.linalg.qr(g)
    return q.reshape(dx, dx, dn).contiguous()


def _environment_matrix(n, seed):
    """Symmetric PSD n x n with eigenvalues (1 + i)^-p, p near 2, and graded eigenvectors."""
    gen = _generator(seed)
    q, _ = torch.linalg.qr(_normal((n, n), gen) * _fall(n, 0.5)[:, None])
    p = 1.9 + 0.2 * float(torch.rand((), generator=gen, device=DEVICE, dtype=torch.float64))
    m = (q * _fall(n, p)) @ q.T
    return (0.5 * (m + m.T)).contiguous()


def _gemm_operands(case, seed):
    gen = _generator(seed)
    return _normal((case["m"], case["k"]), gen), _normal((case["k"], case["n"]), gen)


def _beta(case, seed):
    return case["beta"] + 1e-4 * float(np.random.default_rng(seed).uniform())


def prepare(case, seed):
    kind = case["kind"]
    state = {"case": case, "solver": Solver(0, precision=case["precision"], split_slices=case["slices"])}
    if kind == "gemm":
        state["a"], state["b"] = _gemm_operands(case, seed)
    elif kind == "environment":
        state["t"] = _site_tensor(case["dx"], case["dy"], seed)
    elif kind == "isometry":
        state["m"] = _environment_matrix(case["n"], seed)
    elif kind == "contract":
        state["t"] = _site_tensor(case["dx"], case["dy"], seed)
        state["u"] = _isometry(case["dx"], case["dn"], seed)
    else:
        state["beta"] = _beta(case, seed)
    return state


def run(state):
    case, s = state["case"], state["solver"]
    kind = case["kind"]
    if kind == "gemm":
        return s.gemm(state["a"], state["b"])
    if kind == "environment":
        return s.environment(state["t"])
    if kind == "isometry":
        u, lam, dn = s.isometry(state["m"], case["dcut"])
        return {"u": u, "lam": lam, "dn": dn}
    if kind == "contract":
        return s.contract(state["t"], state["u"])
    s.init_tensor("ising", state["beta"], case["h"])
    s.coarse_grain(case["dcut"], case["nsteps"])
    f, lnz = s.free_energy()
    # the spectrum of the first truncated half-step: later ones depend on the
    # gauge that degenerate levels are left with
    lam = s.spectrum(3 if case["dcut"] < 16 else 5)
    return {"f": f, "lnz": lnz, "spectrum": lam / lam[0]}


# ------------------------------------------------------- work, exact values
def _solve_dims(case):
    """(dx, dy, dn) of every half-step as the x formulas see it."""
    dx = dy = 2
    for k in range(case["nsteps"]):
        a, b = (dx, dy) if k % 2 == 0 else (dy, dx)
        n = min(a * a, case["dcut"])
        yield a, b, n
        if k % 2 == 0:
            dx = n
        else:
            dy = n


def _env_flops(dx, dy):
    # the two Gram products (half of each is enough) and the last product
    return 2.0 * (dx * dy) ** 3 + 2.0 * dx ** 4 * dy ** 2


def _contract_flops(dx, dy, dn):
    return 2.0 * dn * dx ** 3 * dy ** 2 + 2.0 * dn * dx ** 3 * dy ** 3 + 2.0 * dn ** 2 * dx ** 2 * dy ** 2


def _iso_flops(n, dn):
    # a handful of products of M with a block of the kept size
    return 6 * 2.0 * n * n * dn


def work(case):
    kind = case["kind"]
    if kind == "gemm":
        m, n, k = case["m"], case["n"], case["k"]
        return {"bytes": 8.0 * (m * k + k * n + m * n), "flops": 2.0 * m * n * k}
    if kind == "environment":
        dx, dy = case["dx"], case["dy"]
        return {"bytes": 8.0 * ((dx * dy) ** 2 + dx ** 4), "flops": _env_flops(dx, dy)}
    if kind == "isometry":
        n, dn = case["n"], case["dcut"]
        return {"bytes": 8.0 * (n * n + n * dn), "flops": _iso_flops(n, dn)}
    if kind == "contract":
        dx, dy, dn = case["dx"], case["dy"], case["dn"]
        return {"bytes": 8.0 * ((dx * dy) ** 2 + dx * dx * dn + (dn * dy) ** 2),
                "flops": _contract_flops(dx, dy, dn)}
    flops = nbytes = 0.0
    for dx, dy, dn in _solve_dims(case):
        flops += _contract_flops(dx, dy, dn)
        nbytes += 8.0 * ((dx * dy) ** 2 + (dn * dy) ** 2)
        if dn < dx * dx:
            flops += _env_flops(dx, dy) + _iso_flops(dx * dx, dn)
    return {"bytes": nbytes, "flops": flops}


def exact(case, seed):
    kind = case["kind"]
    if kind == "gemm":
        a, b = _gemm_operands(case, seed)
        return a @ b
    if kind == "environment":
        dx, dy = case["dx"], case["dy"]
        t = _site_tensor(dx, dy, seed)
        a = t.permute(0, 3, 1, 2).reshape(dx * dy, dx * dy)     # (j, e), (a, b)
        p = (a @ a.T).reshape(dx, dy, dx, dy)                   # P[j, e, l, f]
        c = t.reshape(dx * dy, dx * dy)                         # (i, e), (c, d)
        q = (c @ c.T).reshape(dx, dy, dx, dy)                   # Q[i, e, k, f]
        left = q.permute(0, 2, 1, 3).reshape(dx * dx, dy * dy)  # (i, k), (e, f)
        right = p.permute(1, 3, 0, 2).reshape(dy * dy, dx * dx)  # (e, f), (j, l)
        m = (left @ right).reshape(dx, dx, dx, dx)              # i, k, j, l
        return m.permute(0, 2, 1, 3).reshape(dx * dx, dx * dx).contiguous()
    if kind == "isometry":
        lam = torch.linalg.eigvalsh(_environment_matrix(case["n"], seed))
        lam = torch.flip(lam, (0,))[:case["dcut"]].cpu().numpy()
        # eigenvectors are fixed up to their signs only
        return {"u": None, "lam": lam, "dn": None}
    if kind == "contract":
        dx, dy, dn = case["dx"], case["dy"], case["dn"]
        t, u = _site_tensor(dx, dy, seed), _isometry(dx, dn, seed)
        out = torch.empty((dn, dy, dn, dy), device=DEVICE, dtype=torch.float64)
        low = t.reshape(dx, dy, dx, dy).permute(1, 0, 2, 3).reshape(dy * dx, dx * dy)   # (c, a), (e, l)
        ub = u.permute(2, 0, 1).reshape(dn * dx, dx)                                    # (i, a), b
        uk = u.reshape(dx * dx, dn)                                                     # (e, d), k
        for j in range(dy):
            top = t[:, j].reshape(dx, dx * dy)                                          # b, (d, c)
            x1 = (ub @ top).reshape(dn, dx, dx, dy).permute(0, 2, 3, 1)                 # i, d, c, a
            x2 = (x1.reshape(dn * dx, dy * dx) @ low).reshape(dn, dx, dx, dy)           # i, d, e, l
            x3 = x2.permute(0, 3, 2, 1).reshape(dn * dy, dx * dx) @ uk                  # (i, l), k
            out[:, j] = x3.reshape(dn, dy, dn).permute(0, 2, 1)
        return out
    return None
