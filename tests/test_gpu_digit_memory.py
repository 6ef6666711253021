"""Scratch of the FP64 digit products: bounded, given up for other buffers, of no effect on results.

An allocator hook that refuses what exceeds a limit stands for a device that is
short of memory.  The digits are then cut in smaller blocks, and their scratch,
which is only kept for the next product, goes when another buffer needs it.
"""
import numpy as np
import pytest

from paper_2306_00358_gb300 import Solver, _lib
from paper_2306_00358_gb300 import serving as sv

pytestmark = pytest.mark.gpu
MIB = 1 << 20


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


class _Limited:
    """Allocations of one context, refused above `limit` live bytes."""

    def __init__(self, torch):
        self.live = self.peak = self.largest = 0
        self.limit = None
        self.sizes = {}

        def alloc(nbytes, stream, user):
            n = int(nbytes)
            if self.limit is not None and self.live + n > self.limit:
                return None
            p = int(torch.cuda.caching_allocator_alloc(n, 0, stream or 0))
            self.sizes[p] = n
            self.live += n
            self.peak = max(self.peak, self.live)
            self.largest = max(self.largest, n)
            return p

        def free(ptr, nbytes, stream, user):
            self.live -= self.sizes.pop(ptr, 0)
            torch.cuda.caching_allocator_delete(ptr)

        self.alloc = _lib.ALLOC_FN(alloc)
        self.free = _lib.FREE_FN(free)


def _solver(mem, **config):
    s = Solver(0, torch_alloc=False, **config)
    s._check(s._lib.trg_set_allocator(s._h, mem.alloc, mem.free, None), "trg_set_allocator")
    return s


def _inputs(torch, d, dn, sectors):
    rng = np.random.default_rng(d)

    def x(*shape):
        i = np.indices(shape)
        weak = (i.sum(0) % 2 == 1) & (i[0] < d // 2)
        return torch.from_numpy(rng.uniform(0.5, 1.0, shape) * np.where(weak, sectors, 1.0)).cuda()

    return x(d, d, d, d), x(d, d, dn)


# 1: nine digits suffice; 2^-24: not for all rows; 2^-80: some elements are left to the pipe
@pytest.mark.parametrize("sectors", [1.0, 2.0 ** -24, 2.0 ** -80])
@pytest.mark.parametrize("room", [0.5, 0.15, 0.06])
def test_less_room_for_the_digits_changes_no_bit(torch, sectors, room):
    d, dn = 32, 31
    t, u = _inputs(torch, d, dn, sectors)
    mem = _Limited(torch)
    with _solver(mem, workspace_bytes=64 * MIB) as s:
        out, m = s.contract(t, u), s.environment(t)
        peak = mem.peak
    digits = mem.largest                 # the largest buffer
    assert digits > 64 * MIB
    tight = _Limited(torch)
    tight.limit = peak - digits + int(room * digits)
    with _solver(tight, workspace_bytes=64 * MIB) as s:
        assert torch.equal(s.contract(t, u), out)
        assert torch.equal(s.environment(t), m)
    assert tight.peak <= tight.limit


def test_scratch_goes_when_another_buffer_needs_the_room(torch):
    t, u = _inputs(torch, 32, 32, 1.0)
    with Solver(0) as s:
        ref = s.environment(t)
    mem = _Limited(torch)
    with _solver(mem, workspace_bytes=64 * MIB) as s:
        s.contract(t, u)
        mem.limit = mem.live + 4 * MIB   # P and Q of the environment take 8 MiB each
        assert torch.equal(s.environment(t), ref)
    assert mem.peak <= mem.limit


def test_digits_stay_within_the_bound(torch):
    t, u = _inputs(torch, 48, 48, 1.0)
    mem = _Limited(torch)
    with _solver(mem, workspace_bytes=300 * MIB) as s:
        s.contract(t, u)
    # flags and marks of the blocks come on top of the digits: a few per cent
    assert mem.largest <= int(300 * MIB * 1.05)


def test_served_result_does_not_depend_on_the_budget(torch):
    spec = sv.Spec(model="ising", beta=0.43, h=1e-3, dcut=32, nsteps=16, precision="fp64")
    with Solver(0) as s:
        s.init_tensor("ising", 0.43, 1e-3)
        s.coarse_grain(32, 16)
        ref = s.free_energy()
    full = sv.solve_bytes(spec, 1 << 30)
    for budget in (full, int(0.85 * full), int(0.7 * full)):
        with sv.Server(0, slots=1, hbm_budget_bytes=budget, workspace_bytes=1 << 30) as server:
            r = server.wait(server.submit(spec))
        assert r["status"] == 0 and (r["f"], r["lnz_per_site"]) == ref, budget
