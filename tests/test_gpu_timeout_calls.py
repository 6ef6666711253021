"""A device wait that runs out is reported by the call that launched the product.

As in test_gpu_timeout.py the epilogue's wait for finished accumulators gets a
1 ns limit, so it runs out while the products it waited for complete on their
own; nothing faults or hangs.  Every call whose products wait on the device
has to say so instead of returning numbers, in both precisions, and the same
context has to give its earlier results again afterwards.
"""
import numpy as np
import pytest

from paper_2306_00358_gb300 import Solver, _lib
from paper_2306_00358_gb300.solver import TRGError

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


def _environment(torch, s, t, u):
    return s.environment(t)


def _contract(torch, s, t, u):
    return s.contract(t, u)


def _isometry(torch, s, t, u):
    # 4096 rows: long enough for the tensor-core form of the FP64 products
    x = t.reshape(4096, -1) * (1.0 + torch.arange(t.numel() // 4096, device="cuda")) ** -1.0
    vec, lam, dn = s.isometry((x @ x.T).contiguous(), 64)
    return torch.from_numpy(lam)


def _solve(torch, s, t, u):
    s.init_tensor("ising", 0.44, 1e-3)
    s.coarse_grain(24, 8)
    return torch.tensor(s.free_energy(), dtype=torch.float64)


def _shard(torch, s, t, u):
    # the first part of a split half-step
    s.init_tensor_raw(t.cpu().numpy(), 1.0)
    slab = torch.zeros(4 * 24 * 24 * t.shape[1], dtype=torch.float64, device="cuda")
    s.shard_begin(24, 0, 4, slab)
    return slab


@pytest.mark.parametrize("precision", ["fp64", "split"])
@pytest.mark.parametrize("call", [_environment, _contract, _isometry, _solve, _shard])
def test_timeout_is_reported_then_the_context_recovers(torch, precision, call):
    rng = np.random.default_rng(11)
    d = 32
    # entries fall off with every leg, as a solve's tensors do
    fall = (1.0 + np.arange(d)) ** -0.75
    t = torch.from_numpy(rng.standard_normal((d, d, d, d)) * np.einsum("i,j,k,l->ijkl", fall, fall, fall, fall)).cuda()
    u = torch.from_numpy(rng.standard_normal((d, d, d))).cuda()
    with Solver(0, precision=precision) as s:
        ref = call(torch, s, t, u)
        s.set_wait_limit(1)
        with pytest.raises(TRGError) as e:
            call(torch, s, t, u)
        assert e.value.status == _lib.TRG_ETIMEOUT
        s.set_wait_limit(0)
    with Solver(0, precision=precision) as s:
        s.set_wait_limit(1)
        with pytest.raises(TRGError) as e:
            call(torch, s, t, u)
        assert e.value.status == _lib.TRG_ETIMEOUT
        s.set_wait_limit(0)
        again = call(torch, s, t, u)
        torch.cuda.synchronize()
        assert torch.equal(again, ref)


def test_timeout_of_a_cubic_lattice_solve(torch):
    with Solver(0, precision="split") as s:
        ref = s.solve3d(0.22, 0.0, 8, 5)
        s.set_wait_limit(1)
        with pytest.raises(TRGError) as e:
            s.solve3d(0.22, 0.0, 8, 5)
        assert e.value.status == _lib.TRG_ETIMEOUT
        s.set_wait_limit(0)
        assert s.solve3d(0.22, 0.0, 8, 5) == ref
