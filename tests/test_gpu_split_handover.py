"""Split contraction: the exponents one product records for the next are those of its output.

The first two products of a contraction record the largest exponent of each row
of their consumer while they store, so the consumer skips a pass.  A chain of
plain products takes its exponents from the FP64 outputs instead; the digits,
and so the results, have to be the same bit for bit.
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


def _chain(torch, s, t, u):
    dx, dy, dn = t.shape[0], t.shape[1], u.shape[2]
    out = torch.empty((dn, dy, dn, dy), device="cuda", dtype=torch.float64)
    ub = u.permute(2, 0, 1).reshape(dn * dx, dx).contiguous()
    low = t.permute(1, 0, 2, 3).reshape(dy * dx, dx * dy).contiguous()
    uk = u.reshape(dx * dx, dn).contiguous()
    for j in range(dy):
        x1 = s.gemm(ub, t[:, j].reshape(dx, dx * dy).contiguous()).reshape(dn, dx, dx, dy)      # i, a, d, c
        x2 = s.gemm(x1.permute(0, 2, 3, 1).reshape(dn * dx, dy * dx).contiguous(), low)         # (i, d), (e, l)
        x2 = x2.reshape(dn, dx, dx, dy).permute(0, 3, 2, 1).reshape(dn * dy, dx * dx)           # (i, l), (e, d)
        out[:, j] = s.gemm(x2.contiguous(), uk).reshape(dn, dy, dn).permute(0, 2, 1)
    return out


# bond dimensions that fill tiles and odd ones; products of one run (K up to 512,
# with an epilogue of their own) and of several
@pytest.mark.parametrize("dx,dy,dn,slices", [(32, 32, 32, 4), (64, 16, 24, 4), (45, 21, 47, 4), (13, 37, 20, 3), (20, 9, 33, 5),
                                             (17, 16, 16, 2)])
@pytest.mark.parametrize("kind", ["plain", "graded"])
def test_contraction_equals_a_chain_of_products(torch, dx, dy, dn, slices, kind):
    rng = np.random.default_rng(dx + dy + dn)
    t, u = rng.standard_normal((dx, dy, dx, dy)), rng.standard_normal((dx, dx, dn))
    if kind == "graded":
        # rows of every size, zero rows, and entries far below their row's largest
        t *= 2.0 ** -rng.integers(0, 60, (dx, dy, dx, 1)) * rng.integers(0, 2, (dx, 1, 1, dy))
        u *= 2.0 ** -rng.integers(0, 90, (1, dx, dn))
        t[dx // 2] = 0.0
        u[:, :, dn - 1] = 0.0
    t, u = torch.from_numpy(t).cuda(), torch.from_numpy(u).cuda()
    with Solver(0, precision="split", split_slices=slices) as s:
        assert torch.equal(s.contract(t, u), _chain(torch, s, t, u))
