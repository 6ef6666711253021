"""Environments that are not finite: the isometry refuses them and the context stays usable.

The Ritz values of such a matrix are NaN.  They are sorted by rank, and the
ranks have to stay a permutation, since they are used as indices.
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


@pytest.mark.parametrize("precision", ["fp64", "split"])
@pytest.mark.parametrize("n,dcut", [(25, 5), (256, 16), (256, 63)])
@pytest.mark.parametrize("value", [float("nan"), float("inf"), float("-inf")])
@pytest.mark.parametrize("where", ["one", "row", "all"])
def test_isometry_of_a_matrix_that_is_not_finite(torch, precision, n, dcut, value, where):
    rng = np.random.default_rng(n)
    x = torch.from_numpy(rng.standard_normal((n, n)) * (1.0 + np.arange(n)) ** -1.0).cuda()
    m = (x @ x.T).contiguous()
    bad = m.clone()
    if where == "one":
        bad[3, 4] = bad[4, 3] = value
    elif where == "row":
        bad[3] = value
        bad[:, 3] = value
    else:
        bad[:] = value
    with Solver(0, precision=precision) as s:
        ref = s.isometry(m, dcut)
        if precision == "fp64":
            with pytest.raises(TRGError) as e:
                s.isometry(bad, dcut)
            assert e.value.status == _lib.TRG_ENUMERIC
        else:
            # the slices hold no infinity or NaN: whatever comes out, the call returns
            try:
                s.isometry(bad, dcut)
            except TRGError as e:
                assert e.status == _lib.TRG_ENUMERIC
        u, lam, dn = s.isometry(m, dcut)
        torch.cuda.synchronize()
        assert dn == ref[2] and torch.equal(u, ref[0]) and np.array_equal(lam, ref[1])
