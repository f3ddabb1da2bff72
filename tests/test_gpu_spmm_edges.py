"""Multi right-hand-side products at the sizes where their paths change: rows
that fit a warp's stage together, alone or not at all, arrays no bulk copy can
read, one or two lane groups per row, strips that straddle a warp's rows,
batches with more and fewer units than the queue has shares."""
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


def check(a, X, Y):
    """Any summation order of n exact products in FP32: within (n + 2) 2^-24 of the sum of their magnitudes."""
    for c in range(X.shape[1]):
        yref, absy = orc.csr_spmv(a.row_ptr, a.col_ind, a.val.astype(np.float32).astype(np.float64),
                                  X[:, c].astype(np.float64))
        tol = (np.diff(a.row_ptr) + 2) * 2.0**-24 * absy
        assert (np.abs(Y[:, c].astype(np.float64) - yref) <= tol).all(), c


def lengths(kind):
    rng = np.random.default_rng(9)
    if kind == "short":  # mean below 8: one lane group per row; empty rows
        return rng.integers(0, 9, 400)
    if kind == "medium":
        return rng.integers(10, 61, 300)
    if kind == "stage_edge":  # rows of exactly the stage, one more, one less, among short ones
        L = rng.integers(0, 20, 200)
        L[[5, 40, 41, 90, 199]] = [704, 705, 703, 352, 5000]
        return L
    return np.full(37, 900)  # no row fits


def convert(b, a, h, offset=0):
    rp, ci = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col_ind).cuda()
    M = b.cmrs_from_csr(rp, ci, torch.from_numpy(a.val.astype(np.float32)).cuda(), a.cols, h, dtype=b.CMRS_F32)
    if offset:  # the same matrix 4 bytes past a 16-byte boundary
        pk = torch.zeros(a.nnz + 8, dtype=torch.int32, device="cuda")[1:1 + a.nnz]
        va = torch.zeros(4 * a.nnz + 32, dtype=torch.uint8, device="cuda")[4:4 + 4 * a.nnz]
        pk.copy_(M.col_packed[:a.nnz])
        va.copy_(M.val[:4 * a.nnz])
        M.col_packed, M.val = pk, va
        M.struct.col_packed, M.struct.val = pk.data_ptr(), va.data_ptr()
    return M


@pytest.mark.parametrize("kind", ["short", "medium", "stage_edge", "long"])
@pytest.mark.parametrize("h", [1, 3, 32])
@pytest.mark.parametrize("k", [1, 2, 4, 8, 12, 32, 36])
@pytest.mark.parametrize("offset", [0, 1])
def test_spmm_paths(b, kind, h, k, offset):
    a = inputs.from_lengths(lengths(kind), 6000, seed=4)
    X = np.random.default_rng(k).standard_normal((a.cols, k)).astype(np.float32)
    M = convert(b, a, h, offset)
    Xd = torch.from_numpy(X).cuda()
    Y = b.cmrs_spmm(M, Xd)
    check(a, X, Y.cpu().numpy())
    Y2 = torch.full_like(Y, float("nan"))
    plan = b.SpmmPlan([M], [Xd], [Y2], work_target=512)
    b.cmrs_spmm_batched(plan)
    b.cmrs_spmm_batched(plan)
    assert torch.equal(Y, Y2)  # the same sums whatever warp takes a row
    plan.close()


def test_spmm_batch_of_many_units(b):
    """More units than shares times blocks, wide and narrow products in turn: every row of every product once."""
    mats, Xs, Ys, As = [], [], [], []
    for i, k in enumerate([32, 32, 8, 1, 16, 4, 2, 32]):
        a = inputs.banded_random(9000 + 17 * i, 300, 10, 60, seed=i)
        M = convert(b, a, [1, 2, 4][i % 3])
        X = np.random.default_rng(i).standard_normal((a.cols, k)).astype(np.float32)
        As.append(a)
        mats.append(M)
        Xs.append(torch.from_numpy(X).cuda())
        Ys.append(torch.full((a.rows, k), float("nan"), device="cuda"))
    plan = b.SpmmPlan(mats, Xs, Ys, work_target=256)
    assert plan.info()["units"] > 8 * 152 * 2
    b.cmrs_spmm_batched(plan)
    for a, M, X, Y in zip(As, mats, Xs, Ys):
        assert torch.equal(Y, b.cmrs_spmm(M, X))
        check(a, X.cpu().numpy()[:, :1], Y.cpu().numpy()[:, :1])
    plan.close()
