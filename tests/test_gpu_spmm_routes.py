"""Products by both ways, staged and walked: the same bits whichever way a row goes, and within the bound of any order."""
import numpy as np
import pytest
import torch

import oracle as orc
from paper_1203_2946_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1203_2946_gb300 import build
    build.build()
    from paper_1203_2946_gb300 import binding
    return binding


def convert(b, a, h):
    return b.cmrs_from_csr(torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col_ind).cuda(),
                           torch.from_numpy(a.val.astype(np.float32)).cuda(), a.cols, h, dtype=b.CMRS_F32)


# rows of 0..4, of 8 to 30, of 60..90 and of 350..500 entries, for a product alone; each beside a wide and a narrow
# product of another matrix, which takes the batch the other way
@pytest.mark.parametrize("lo,hi,rows", [(0, 4, 3000), (8, 30, 1500), (60, 90, 500), (350, 500, 120)])
@pytest.mark.parametrize("h", [1, 3, 16])
@pytest.mark.parametrize("k", [1, 2, 3, 4, 8, 16, 64])
def test_same_sums_either_way(b, lo, hi, rows, h, k):
    rng = np.random.default_rng(lo + h)
    a = inputs.from_lengths(rng.integers(lo, hi + 1, rows), 4000, seed=6)
    X = rng.standard_normal((a.cols, k)).astype(np.float32)
    M, Xd = convert(b, a, h), torch.from_numpy(X).cuda()
    Y = b.cmrs_spmm(M, Xd, torch.full((rows, k), float("nan"), device="cuda"))
    for c in (0, k - 1):
        yref, absy = orc.csr_spmv(a.row_ptr, a.col_ind, a.val.astype(np.float32).astype(np.float64), X[:, c].astype(np.float64))
        tol = (np.diff(a.row_ptr) + 2) * 2.0**-24 * absy  # any order of n exact products
        assert (np.abs(Y[:, c].cpu().numpy().astype(np.float64) - yref) <= tol).all()
    other = convert(b, inputs.banded_random(40_000, 200, 10, 60, seed=1), 1)
    for ko in (1, 8):
        Xo = torch.ones((other.cols, ko), device="cuda")
        Ys = [torch.full((rows, k), float("nan"), device="cuda"), torch.empty((other.rows, ko), device="cuda")]
        plan = b.SpmmPlan([M, other], [Xd, Xo], Ys, work_target=1024)
        b.cmrs_spmm_batched(plan)
        b.cmrs_spmm_batched(plan)
        assert torch.equal(Ys[0], Y)
        plan.close()
