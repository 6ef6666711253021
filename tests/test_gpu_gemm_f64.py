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
