"""Split contraction: short products (K = Dx up to 512 in one run) store their
results with exponents added to the high words.

Scaling column i of U by 2^s_i scales the row exponents of every product that
holds i and nothing else, so Tx[i, j, k, l] scales by 2^(s_i + s_k) bit for bit.
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


def _inputs(dx, dy, dn):
    rng = np.random.default_rng(100 * dx + 10 * dy + dn)
    t = rng.standard_normal((dx, dy, dx, dy))
    t[dx // 2] = 0.0            # exact zeros among the results
    t[:, :, :, dy - 1] = 0.0
    return t, rng.standard_normal((dx, dx, dn))


def _run(torch, t, u, slices):
    with Solver(0, precision="split", split_slices=slices) as s:
        return s.contract(torch.from_numpy(t).cuda(), torch.from_numpy(u).cuda()).cpu().numpy()


# ragged rows and columns of the 128 x 128 tile, K below one stage and above it
@pytest.mark.parametrize("dx,dy,dn", [(7, 5, 3), (16, 16, 16), (19, 33, 21), (40, 12, 35)])
@pytest.mark.parametrize("slices", [2, 3, 4, 5])
def test_scaling_u_scales_the_result_exactly(torch, dx, dy, dn, slices):
    t, u = _inputs(dx, dy, dn)
    s = (np.arange(dn) * 37) % 601 - 300
    base = _run(torch, t, u, slices)
    out = _run(torch, t, np.ldexp(u, s), slices)
    assert np.array_equal(out, np.ldexp(base, s[:, None, None, None] + s[None, None, :, None]))
    # each product is off by at most (S + 2) K 2^(1 - 8 S) of its largest entries
    eps = (slices + 2) * 2.0 ** (1 - 8 * slices)
    tm, um = np.abs(t).max(), np.abs(u).max()
    x1, e1 = dx * um * tm, eps * dx * um * tm
    x2, e2 = dx * dy * x1 * tm, dx * dy * tm * (e1 + eps * x1)
    bound = dx * dx * um * (e2 + eps * x2)
    x = np.einsum("abi,bjdc->ijdac", u, t, optimize=True)
    ref = np.einsum("ijdac,acel,edk->ijkl", x, t, u, optimize=True)
    assert np.abs(base - ref).max() <= bound


# results below the normal range come out as zero, the others are untouched
def test_results_below_the_normal_range(torch):
    t, u = _inputs(19, 17, 12)
    s = np.zeros(12, dtype=int)
    s[[2, 7]] = [-1024, -1030]
    base = _run(torch, t, u, 4)
    out = _run(torch, t, np.ldexp(np.sign(u) * (np.abs(u) + 4.0), s), 4)
    ref = _run(torch, t, np.sign(u) * (np.abs(u) + 4.0), 4)
    keep = np.ones(12, dtype=bool)
    keep[[2, 7]] = False
    assert np.array_equal(out[keep][:, :, keep], ref[keep][:, :, keep])
    assert np.abs(out[~keep]).max() <= 2.0 ** -1000 and np.abs(out[:, :, ~keep]).max() <= 2.0 ** -1000
    assert np.isfinite(base).all()
