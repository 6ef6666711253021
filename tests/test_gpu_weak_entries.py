"""FP64 products keep the accuracy of entries far below the largest of their row and column.

The tensor-core form of a large FP64 product cuts its operands to fixed point
relative to the largest entry of each row and column, so an element whose sum
|a||b| lies far below the product of those scales takes the FP64 pipe instead.
Whatever the form, an element is within (K + 1) 2^-53 |A||B| of the exact
product; two such results may differ by twice that.
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


def _contract(torch, t, u):
    x1 = torch.einsum("abi,bjdc->ijdac", u, t)
    x2 = torch.einsum("ijdac,acel->ijdel", x1, t)
    return torch.einsum("ijdel,edk->ijkl", x2, u)


def _environment(torch, t):
    dx, dy = t.shape[0], t.shape[1]
    a = t.permute(0, 3, 1, 2).reshape(dx * dy, dx * dy)
    c = t.reshape(dx * dy, dx * dy)
    p, q = (a @ a.T).reshape(dx, dy, dx, dy), (c @ c.T).reshape(dx, dy, dx, dy)
    left = q.permute(0, 2, 1, 3).reshape(dx * dx, dy * dy)
    right = p.permute(1, 3, 0, 2).reshape(dy * dy, dx * dx)
    return (left @ right).reshape(dx, dx, dx, dx).permute(0, 2, 1, 3).reshape(dx * dx, dx * dx)


def _sectors(torch, rng, shape, eps):
    """Even and odd index sums, coupled by eps."""
    odd = np.indices(shape).sum(0) % 2
    x = rng.uniform(0.5, 1.0, shape) * rng.choice([-1.0, 1.0], shape) * np.where(odd, eps, 1.0)
    return torch.from_numpy(x).cuda()


def _scattered(torch, rng, shape, span):
    """Exponents spread evenly over `span` powers of two, a third of the entries zero."""
    x = rng.uniform(0.5, 1.0, shape) * rng.choice([-1.0, 1.0, 0.0], shape) * 2.0 ** -rng.uniform(0.0, span, shape)
    return torch.from_numpy(x).cuda()


def _check_contract(torch, t, u):
    dx, dy, dn = t.shape[0], t.shape[1], u.shape[2]
    with Solver(0) as s:
        out = s.contract(t, u)
    bound = 2.0 * (dx + 1 + dx * dy + 1 + dx * dx + 1) * 1.01 * 2.0 ** -53 * _contract(torch, t.abs(), u.abs())
    assert bool(((out - _contract(torch, t, u)).abs() <= bound).all())


def _check_environment(torch, t):
    dx, dy = t.shape[0], t.shape[1]
    with Solver(0) as s:
        m = s.environment(t)
    bound = 2.0 * (2 * (dx * dy + 1) + dy * dy + 1) * 1.01 * 2.0 ** -53 * _environment(torch, t.abs())
    assert bool(((m - _environment(torch, t)).abs() <= bound).all())


# sums at, just above and far below what 15 digits reach, each with remainders
# of the 128 x 32 tiles; 48: long enough to look for the nine-digit form
@pytest.mark.parametrize("eps", [2.0 ** -50, 2.0 ** -58, 2.0 ** -61, 2.0 ** -90, 2.0 ** -125, 2.0 ** -200])
@pytest.mark.parametrize("dx,dy,dn", [(16, 16, 16), (24, 24, 24), (27, 22, 31), (48, 20, 33)])
def test_contraction_of_hardly_coupled_sectors(torch, eps, dx, dy, dn):
    rng = np.random.default_rng(dx)
    _check_contract(torch, _sectors(torch, rng, (dx, dy, dx, dy), eps), _sectors(torch, rng, (dx, dx, dn), eps))


@pytest.mark.parametrize("span", [40.0, 150.0])
@pytest.mark.parametrize("dx,dy,dn", [(24, 24, 24), (29, 17, 19)])
def test_contraction_of_scattered_exponents(torch, span, dx, dy, dn):
    rng = np.random.default_rng(int(span))
    _check_contract(torch, _scattered(torch, rng, (dx, dy, dx, dy), span), _scattered(torch, rng, (dx, dx, dn), span))


# P and Q in one launch (up to 640 rows) and each alone
@pytest.mark.parametrize("eps", [2.0 ** -58, 2.0 ** -61, 2.0 ** -125])
@pytest.mark.parametrize("dx,dy", [(16, 16), (24, 22), (19, 33), (33, 32)])
def test_environment_of_hardly_coupled_sectors(torch, eps, dx, dy):
    rng = np.random.default_rng(dx + dy)
    _check_environment(torch, _sectors(torch, rng, (dx, dy, dx, dy), eps))


@pytest.mark.parametrize("dx,dy", [(24, 22), (33, 32)])
def test_environment_of_scattered_exponents(torch, dx, dy):
    rng = np.random.default_rng(dx + dy)
    _check_environment(torch, _scattered(torch, rng, (dx, dy, dx, dy), 100.0))


# one entry of a row 2^-70 and 2^-300 below the others, and alone in its column
@pytest.mark.parametrize("small", [2.0 ** -70, 2.0 ** -300])
@pytest.mark.parametrize("at", [(0, 0, 0, 0), (23, 23, 23, 23), (5, 17, 11, 2)])
def test_a_single_small_entry(torch, small, at):
    rng = np.random.default_rng(3)
    d = 24
    t = rng.uniform(0.5, 1.0, (d, d, d, d))
    u = rng.uniform(0.5, 1.0, (d, d, d))
    t[at[0]] = 0.0
    t[:, :, at[2], at[3]] = 0.0
    t[at] = small
    t, u = torch.from_numpy(t).cuda(), torch.from_numpy(u).cuda()
    _check_contract(torch, t, u)
    _check_environment(torch, t)
