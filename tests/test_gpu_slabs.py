"""An element of an FP64 contraction has the same bits whatever slab it is computed in.

A contraction runs in slices of j sized to the workspace, and over ranks each
takes some j's.  Its products are then slabs of whole ones of other sizes, and
how they are computed (FP64 pipe or digits, nine digits or fifteen, K in parts)
must not depend on the slab, nor on what the other rows of it hold.
"""
import numpy as np
import pytest

from paper_2306_00358_gb300 import Solver, sharding

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def torch():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    return torch


def _tensor(d, dy, kind):
    rng = np.random.default_rng(d + dy)
    t = rng.uniform(0.5, 1.0, (d, dy, d, dy))
    odd = np.indices(t.shape).sum(0) % 2
    weak = np.where(odd, 2.0 ** -20, 1.0)
    gone = np.where(odd, 2.0 ** -80, 1.0)
    if kind == "plain":
        return t
    if kind == "weak":
        return t * weak
    # by j: slices that nine digits suffice for, that need fifteen, and that
    # are left to the pipe in part
    j = np.arange(dy).reshape(1, dy, 1, 1)
    return t * np.where(j % 3 == 0, 1.0, np.where(j % 3 == 1, weak, gone))


def _isometry(d, dn):
    return np.random.default_rng(d).uniform(0.5, 1.0, (d, d, dn))


@pytest.mark.parametrize("kind", ["plain", "weak", "mixed"])
@pytest.mark.parametrize("dx,dy,dn", [(12, 12, 12), (24, 24, 24), (33, 20, 25), (32, 40, 32)])
def test_contraction_in_slices_of_any_size(torch, dx, dy, dn, kind):
    t = torch.from_numpy(_tensor(dx, dy, kind)).cuda()
    u = torch.from_numpy(_isometry(dx, dn)).cuda()
    with Solver(0) as s:
        whole = s.contract(t, u)
    per_j = 2 * dn * dx * dx * dy * 8
    for jb in (1, 2, 5):
        with Solver(0, workspace_bytes=jb * per_j) as s:
            assert torch.equal(s.contract(t, u), whole), jb


@pytest.mark.parametrize("kind", ["plain", "weak", "mixed"])
@pytest.mark.parametrize("world", [2, 5, 24])
def test_split_half_step_equals_the_unsplit_one(torch, world, kind):
    d, dcut = 24, 24
    fall = (1.0 + np.arange(d)) ** -0.5
    t = _tensor(d, d, kind) * np.einsum("i,j,k,l->ijkl", fall, fall, fall, fall)
    with Solver(0) as s:
        s.init_tensor_raw(t, 1.0)
        s.coarse_grain(dcut, 1)
        ref = s.tensor()
    rows = sharding.slab_rows(d, world)
    slabs = []
    with Solver(0) as s:
        for j0, j1 in sharding.j_ranges(d, world):
            s.init_tensor_raw(t, 1.0)
            slab = torch.zeros(sharding.slab_elems(rows, dcut, d), dtype=torch.float64, device="cuda")
            assert s.shard_begin(dcut, j0, j1, slab) == dcut
            slabs.append(slab)
        s.init_tensor_raw(t, 1.0)
        s.shard_begin(dcut, 0, 0, slabs[0])
        s.shard_finish(torch.cat(slabs), world * rows)
        np.testing.assert_array_equal(s.tensor(), ref)


def test_split_solve_equals_the_unsplit_one(torch):
    args = dict(model="ising", beta=0.43, h=1e-3)
    with Solver(0) as s:
        s.init_tensor(**args)
        s.coarse_grain(24, 12)
        f, ref = s.free_energy(), s.tensor()
    world = 4
    ranks = [Solver(0) for _ in range(world)]
    for s in ranks:
        s.init_tensor(**args)
    for _ in range(12):
        nj = ranks[0].shard_extent()
        rows = sharding.slab_rows(nj, world)
        parts, dn = [], 0
        for s, (j0, j1) in zip(ranks, sharding.j_ranges(nj, world)):
            slab = torch.zeros(sharding.slab_elems(rows, 24, nj), dtype=torch.float64, device="cuda")
            dn = s.shard_begin(24, j0, j1, slab)
            parts.append(slab[:sharding.slab_elems(rows, dn, nj)])
        for s in ranks:
            s.shard_finish(torch.cat(parts), world * rows)
    for s in ranks:
        assert s.free_energy() == f
        np.testing.assert_array_equal(s.tensor(), ref)
        s.close()
