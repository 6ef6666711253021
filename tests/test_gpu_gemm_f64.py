"""FP64 products over the output tiles the size rule picks, against torch FP64.

Both sides sum K rounded products in some order, so each is within
(K + 1) 2^-53 |A||B| of the exact product, element for element (the standard
bound of a length-K dot product); they may differ by twice that.
"""
import numpy as np
import pytest

from paper_2306_00358_gb300 import Solver

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


def _close(torch, c, a, b):
    k = a.shape[1]
    bound = 2.0 * (k + 1) * 2.0 ** -53 * (a.abs() @ b.abs())
    assert bool(((c - a @ b).abs() <= bound).all())


# 8 x 8 tiles (one output, ragged edges, split K), 16, 32 and 64 wide ones,
# each with remainders in M, N and K
@pytest.mark.parametrize("m,n,k", [(1, 1, 1), (9, 7, 65), (96, 80, 72), (256, 40, 256), (40, 40, 3000),
                                   (257, 41, 1000), (513, 200, 129), (700, 650, 33), (1100, 1030, 70), (3, 2000, 17)])
def test_product_matches_torch(torch, m, n, k):
    rng = np.random.default_rng(m + n + k)
    a = torch.from_numpy(rng.standard_normal((m, k))).cuda()
    b = torch.from_numpy(rng.standard_normal((k, n))).cuda()
    with Solver(0) as s:
        _close(torch, s.gemm(a, b), a, b)


# the Gram products compute the tiles on and above the diagonal and mirror
# the others: P and Q of a (dx, dy) tensor are (dx dy) square
@pytest.mark.parametrize("dx,dy", [(1, 5), (3, 3), (9, 8), (13, 17), (24, 22), (33, 32)])
def test_environment_matches_torch(torch, dx, dy):
    rng = np.random.default_rng(100 * dx + dy)
    t = torch.from_numpy(rng.standard_normal((dx, dy, dx, dy))).cuda()
    with Solver(0) as s:
        m = s.environment(t)

    def env(t):
        a = t.permute(0, 3, 1, 2).reshape(dx * dy, dx * dy)
        c = t.reshape(dx * dy, dx * dy)
        p = (a @ a.T).reshape(dx, dy, dx, dy)
        q = (c @ c.T).reshape(dx, dy, dx, dy)
        left = q.permute(0, 2, 1, 3).reshape(dx * dx, dy * dy)
        right = p.permute(1, 3, 0, 2).reshape(dy * dy, dx * dx)
        return (left @ right).reshape(dx, dx, dx, dx).permute(0, 2, 1, 3).reshape(dx * dx, dx * dx)

    # three products in a row, of lengths dx dy (twice) and dy dy, on each side
    bound = 2.0 * (2 * (dx * dy + 1) + dy * dy + 1) * 1.01 * 2.0 ** -53 * env(t.abs())
    assert bool(((m - env(t)).abs() <= bound).all())


def _contract(torch, t, u):
    # Tx[i,j,k,l] = sum U[a,b,i] t[b,j,d,c] t[a,c,e,l] U[e,d,k], step by step
    x1 = torch.einsum("abi,bjdc->ijdac", u, t)
    x2 = torch.einsum("ijdac,acel->ijdel", x1, t)
    return torch.einsum("ijdel,edk->ijkl", x2, u)


# large enough for the tensor-core form: remainders of the 128 x 64 tile, of
# the 32-deep stages and the 128-deep exact runs; 32: the row-wise stores.
# The tensor-core form is off by at most 2^-53 |C| + 10 K 2^-64 times the
# largest entries of the row and the column of each product, for entries of
# like size far below the chain bound of test_product_matches_torch.
@pytest.mark.parametrize("dx,dy,dn", [(16, 17, 15), (20, 13, 33), (24, 24, 24), (27, 21, 11), (32, 32, 32)])
@pytest.mark.parametrize("ws", [0, 40_000_000])
def test_contraction_matches_torch(torch, dx, dy, dn, ws):
    rng = np.random.default_rng(dx * dy + dn)
    t = torch.from_numpy(rng.standard_normal((dx, dy, dx, dy))).cuda()
    u = torch.from_numpy(rng.standard_normal((dx, dx, dn))).cuda()
    with Solver(0, workspace_bytes=ws) as s:
        out = s.contract(t, u)
    bound = 2.0 * (dx + 1 + dx * dy + 1 + dx * dx + 1) * 1.01 * 2.0 ** -53 * _contract(torch, t.abs(), u.abs())
    assert bool(((out - _contract(torch, t, u)).abs() <= bound).all())


# nearly decoupled sectors (even and odd index sums, coupled by eps): sums of
# products far below the largest ones keep their own accuracy.  0: the odd sums
# are exact zeros; 2^-4: all sums are of like size.
@pytest.mark.parametrize("eps", [0.0, 2.0 ** -70, 2.0 ** -30, 2.0 ** -9, 2.0 ** -4])
@pytest.mark.parametrize("dx,dy,dn", [(16, 16, 16), (24, 24, 24), (27, 22, 31)])
def test_contraction_of_weakly_coupled_sectors(torch, eps, dx, dy, dn):
    rng = np.random.default_rng(dx)

    def graded(*shape):
        odd = np.indices(shape).sum(0) % 2
        x = rng.uniform(0.5, 1.0, shape) * rng.choice([-1.0, 1.0], shape) * np.where(odd, eps, 1.0)
        return torch.from_numpy(x).cuda()

    t, u = graded(dx, dy, dx, dy), graded(dx, dx, dn)
    with Solver(0) as s:
        out = s.contract(t, u)
    bound = 2.0 * (dx + 1 + dx * dy + 1 + dx * dx + 1) * 1.01 * 2.0 ** -53 * _contract(torch, t.abs(), u.abs())
    assert bool(((out - _contract(torch, t, u)).abs() <= bound).all())


# operands outside the digits' range take the FP64 pipe
@pytest.mark.parametrize("scale", [2.0 ** 420, 2.0 ** -420, 2.0 ** -480])
def test_contraction_outside_the_digit_range(torch, scale):
    rng = np.random.default_rng(5)
    d = 24
    t = torch.from_numpy(rng.standard_normal((d, d, d, d))).cuda()
    u = torch.from_numpy(rng.standard_normal((d, d, d))).cuda()
    with Solver(0) as s:
        out = s.contract(t * scale, u)
    k = d + 1 + 2 * (d * d + 1)
    bound = 2.0 * k * 1.01 * 2.0 ** -53 * _contract(torch, t.abs(), u.abs())
    assert bool(((out / scale / scale - _contract(torch, t, u)).abs() <= bound).all())


@pytest.mark.parametrize("value", [float("inf"), float("-inf"), float("nan")])
def test_contraction_carries_infinities_and_nan(torch, value):
    rng = np.random.default_rng(6)
    d = 24
    t = torch.from_numpy(rng.standard_normal((d, d, d, d))).cuda()
    u = torch.from_numpy(rng.standard_normal((d, d, d))).cuda()
    t[3, 4, 5, 6] = value
    with Solver(0) as s:
        out = s.contract(t, u)
    ref = _contract(torch, t, u)
    assert bool((torch.isnan(out) == torch.isnan(ref)).all())
    assert bool((torch.isinf(out) == torch.isinf(ref)).all())


# P and Q share a launch, and its fallback
@pytest.mark.parametrize("value", [float("inf"), float("nan")])
def test_environment_carries_infinities_and_nan(torch, value):
    rng = np.random.default_rng(7)
    dx, dy = 24, 22
    t = torch.from_numpy(rng.standard_normal((dx, dy, dx, dy))).cuda()
    t[3, 4, 5, 6] = value
    with Solver(0) as s:
        m = s.environment(t)
    a = t.permute(0, 3, 1, 2).reshape(dx * dy, dx * dy)
    c = t.reshape(dx * dy, dx * dy)
    p, q = (a @ a.T).reshape(dx, dy, dx, dy), (c @ c.T).reshape(dx, dy, dx, dy)
    ref = torch.einsum("iekf,jelf->ijkl", q, p).reshape(dx * dx, dx * dx)
    assert bool((torch.isnan(m) == torch.isnan(ref)).all())
    assert bool((torch.isinf(m) == torch.isinf(ref)).all())


@pytest.mark.parametrize("zero_rows", [True, False])
def test_environment_of_a_sparse_tensor(torch, zero_rows):
    """Zero rows and columns (exponent field 0) and entries 2^-70 below the largest."""
    rng = np.random.default_rng(8)
    d = 24
    t = rng.standard_normal((d, d, d, d))
    if zero_rows:
        t[5] = 0.0
        t[:, 7] = 0.0
    t[9] *= 2.0 ** -70
    t = torch.from_numpy(t).cuda()
    with Solver(0) as s:
        m = s.environment(t)
    a = t.permute(0, 3, 1, 2).reshape(d * d, d * d)
    c = t.reshape(d * d, d * d)
    p, q = (a @ a.T).reshape(d, d, d, d), (c @ c.T).reshape(d, d, d, d)
    ref = torch.einsum("iekf,jelf->ijkl", q, p).reshape(d * d, d * d)
    # of the largest element: three products, each within (K + 1) 2^-53 on both sides
    assert float((m - ref).abs().max()) <= 2.0 * 3 * (d * d + 1) * 2.0 ** -53 * float(ref.abs().max())
