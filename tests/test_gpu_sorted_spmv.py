"""SpMV on column-sorted strips at the sizes where its paths change: whole
strips per warp (heights that divide 32 and heights that do not), one and two
lanes per row, units longer than the stage, rows longer than the list, empty
rows, arrays no bulk copy can read; matrices large enough for the mapping and
small ones, which keep Algorithm 1."""
import functools

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


def lengths(kind):
    """About 1,000 rows of a kind, or (large_*) 45,000 to 230,000 of them: past the fewest units of the mapping."""
    rng = np.random.default_rng(12)
    if kind.startswith("large_"):
        L = lengths(kind[6:])
        return np.tile(L, {"short": 45, "skewed": 45, "regular": 230, "two": 120}[kind[6:]])
    if kind == "short":
        return rng.integers(0, 9, 1003)
    if kind == "regular":  # mean 27: one lane per row
        return rng.integers(25, 30, 997)
    if kind == "two":  # mean 40
        return rng.integers(20, 61, 901)
    if kind == "four":  # mean 90
        return rng.integers(60, 121, 500)
    if kind == "long":  # no mapping but Algorithm 1
        return rng.integers(100, 160, 200)
    L = rng.integers(0, 12, 1200)  # skewed: a list too short, a stage too small, beside units that fit
    L[[3, 40, 41, 700, 1199]] = [60, 17, 18, 5000, 900]
    L[200:300] = 0
    return L


@functools.lru_cache(maxsize=None)
def matrix(kind):
    L = lengths(kind)
    if not kind.startswith("large_"):
        return inputs.from_lengths(L, 7000, seed=3)
    # one column drawn in each of a row's equal strata: distinct and increasing
    row = np.repeat(np.arange(L.size), L)
    j = np.arange(row.size) - np.repeat(np.cumsum(L) - L, L)
    rng = np.random.default_rng(5)
    lo, hi = j * 7000 // L[row], (j + 1) * 7000 // L[row]
    col = (lo + rng.random(row.size) * (hi - lo)).astype(np.int32)
    rp = np.concatenate([[0], np.cumsum(L)]).astype(np.int32)
    return inputs.CSR(L.size, 7000, rp, col, rng.uniform(-1, 1, row.size), kind)


@pytest.mark.parametrize("kind", ["short", "regular", "two", "four", "long", "skewed", "large_short", "large_skewed",
                                  "large_regular", "large_two"])
@pytest.mark.parametrize("h", [1, 2, 3, 4, 6, 8, 12, 16, 17, 32])
@pytest.mark.parametrize("dtype", [0, 1, 2, 3])
def test_sorted_spmv(b, kind, h, dtype):
    a = matrix(kind)
    rp, ci = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col_ind).cuda()
    M = b.cmrs_from_csr(rp, ci, torch.from_numpy(a.val).cuda(), a.cols, h, flags=b.CMRS_SORTED, dtype=dtype)
    x = inputs.uniform_vector(a.cols, 5)
    x = x if dtype == 0 else x.astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    y = b.cmrs_spmv(M, xd, torch.full((a.rows,), float("nan"), dtype=xd.dtype, device="cuda"))
    b.cmrs_spmv_check(M)
    vq = a.val if dtype == 0 else orc.decode(orc.encode(a.val, dtype), dtype, a.nnz)
    yref, absy = orc.csr_spmv(a.row_ptr, a.col_ind, vq, x.astype(np.float64))
    # FP64: the library's bar; FP32 accumulation: any order of n exact products
    tol = 1e-12 * absy if dtype == 0 else (np.diff(a.row_ptr) + 2) * 2.0**-24 * absy
    assert (np.abs(y.cpu().numpy().astype(np.float64) - yref) <= tol).all()
    # the row map writes the same sums elsewhere; repeated calls are bit-identical
    perm = torch.from_numpy(np.random.default_rng(0).permutation(a.rows).astype(np.int32)).cuda()
    z = b.cmrs_spmv_rows(M, xd, perm)
    assert torch.equal(z[perm.long()], y)
    if dtype == 1:  # 4 bytes past a 16-byte boundary: accepted as before, by Algorithm 1
        pk = torch.zeros(a.nnz + 8, dtype=torch.int32, device="cuda")[1:1 + a.nnz]
        pk.copy_(M.col_packed[:a.nnz])
        M.col_packed = pk
        M.struct.col_packed = pk.data_ptr()
        y2 = b.cmrs_spmv(M, xd).cpu().numpy().astype(np.float64)
        assert (np.abs(y2 - yref) <= tol).all()
