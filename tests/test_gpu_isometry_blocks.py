"""The subspace iteration at the edges of its kernels' block sizes.

Cholesky-QR works on m = min(n, Dcut + 24, 112) columns (odd and even, fewer
than a warp, the largest) and on blocks of 8, 16 or 32 rows by n.  FP64 solves
stop at a Ritz residual of 1e-12 theta_1, so the returned pairs satisfy
|M u - lambda u| <= 1e-12 lambda_1 to rounding, and U is orthonormal to
rounding (m products of unit vectors of length n).
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


def _matrix(torch, n, rank, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    q, _ = torch.linalg.qr(torch.randn((n, n), generator=gen, device="cuda", dtype=torch.float64))
    lam = (1.0 + torch.arange(n, device="cuda", dtype=torch.float64)) ** -3.0
    lam[rank:] = 0.0
    m = (q * lam) @ q.T
    return (0.5 * (m + m.T)).contiguous(), lam


# m = n odd and even, m odd, m = 2 warps + 1, the largest block, and row
# counts on both sides of the 8-, 16- and 32-row blocks (152 SMs) with remainders
@pytest.mark.parametrize("n,dcut", [(3, 1), (4, 2), (25, 1), (30, 3), (64, 41), (150, 88), (160, 111), (1215, 16),
                                    (1217, 17), (2437, 9)])
def test_isometry_pairs(torch, n, dcut):
    m, lam = _matrix(torch, n, n, n + dcut)
    with Solver(0) as s:
        u, got, dn = s.isometry(m, dcut)
    assert dn == dcut
    eps = 2.0 ** -53
    u = u.contiguous()
    eye = torch.eye(dn, device="cuda", dtype=torch.float64)
    assert float((u.T @ u - eye).abs().max()) <= 64 * n ** 0.5 * eps
    got = torch.from_numpy(got).cuda()
    assert float((got - lam[:dn]).abs().max()) <= 2e-12
    res = (m @ u - u * got).norm(dim=0)
    assert float(res.max()) <= 2e-12


# fewer positive eigenvalues than columns: dependent columns are replaced
@pytest.mark.parametrize("n,dcut,rank", [(100, 20, 7), (300, 33, 33), (1300, 16, 5)])
def test_isometry_of_a_rank_deficient_matrix(torch, n, dcut, rank):
    m, lam = _matrix(torch, n, rank, n + rank)
    with Solver(0) as s:
        u, got, dn = s.isometry(m, dcut)
    u = u.contiguous()
    assert float((u.T @ u - torch.eye(dn, device="cuda", dtype=torch.float64)).abs().max()) <= 1e-12
    assert float((torch.from_numpy(got).cuda() - lam[:dn]).abs().max()) <= 2e-12
