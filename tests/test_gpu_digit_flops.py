"""The profile books the digit products that were computed, 45 or 120 for each product.

Which of the two a row takes is decided on the device.
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


def _digit_products(torch, weak_j):
    """Digit products per product of a contraction whose upper tensor has weak couplings for those j."""
    d = 32
    rng = np.random.default_rng(d)
    odd = np.indices((d, d, d, d)).sum(0) % 2
    t = rng.uniform(0.5, 1.0, odd.shape)
    j = np.arange(d).reshape(1, d, 1, 1)
    t = np.where((odd == 1) & (j < weak_j), 2.0 ** -30, 1.0) * t
    u = np.where(np.indices((d, d, d)).sum(0) % 2 == 1, 2.0 ** -30 if weak_j == d else 1.0, 1.0) * rng.uniform(0.5, 1.0, (d, d, d))
    with Solver(0) as s:
        s.profile(True)
        s.contract(torch.from_numpy(t).cuda(), torch.from_numpy(u).cuda())
        ph = s.phase_stats()["mma"]
        again = s.phase_stats()["mma"]
        assert again["mma_flops"] == ph["mma_flops"]
        s.profile(False)
    return ph["mma_flops"] / ph["flops"]


def test_digit_products_of_a_contraction(torch):
    # every length here is a multiple of the 32 that K is padded to
    assert _digit_products(torch, 32) == pytest.approx(120.0, rel=1e-9)
    # the D^7 product, 15/16 of the work, takes nine digits
    assert 45.0 <= _digit_products(torch, 0) <= 45.0 + 75.0 / 8
