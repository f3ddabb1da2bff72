"""MERGE by every tile set it launches: the sizes either side of a wave of CTAs, where the FP32-accumulated forms change
between 11 and 13 entries a thread, and long rows over several tiles a CTA."""
import functools

import numpy as np
import pytest
import torch

import oracle as orc
from paper_1203_2946_gb300 import inputs

pytestmark = pytest.mark.gpu

WAVE = 6 * 128  # entries a thread x this x SMs: a wave of CTAs on short rows


@pytest.fixture(scope="module")
def b():
    from paper_1203_2946_gb300 import build
    build.build()
    from paper_1203_2946_gb300 import binding
    return binding


@functools.lru_cache(maxsize=None)
def matrix(waves11, mean):
    """Rows of 0 to 2 x mean entries, so many of them as fill the given number of waves at 11 entries a thread."""
    nnz = int(waves11 * 11 * WAVE * torch.cuda.get_device_properties(0).multi_processor_count)
    rng = np.random.default_rng(6)
    L = rng.integers(0, 2 * mean + 1, nnz // mean)
    L[[5, 6]] = [40_000, 0]  # a row over many tiles
    row = np.repeat(np.arange(L.size), L)
    col = rng.integers(0, 60_000, row.size).astype(np.int32)
    rp = np.concatenate([[0], np.cumsum(L)]).astype(np.int32)
    return inputs.CSR(L.size, 60_000, rp, col, rng.uniform(-1, 1, row.size), "tiles")


# short rows: one wave (11 entries), one with 13 where 11 need two, two of 11, three and more of 13; long rows
@pytest.mark.parametrize("waves11,mean", [(0.4, 4), (1.09, 4), (1.5, 4), (2.8, 4), (2.5, 20)])
@pytest.mark.parametrize("h", [1, 5, 32])
@pytest.mark.parametrize("dtype", [0, 1, 2, 3])
def test_merge_tiles(b, waves11, mean, h, dtype):
    a = matrix(waves11, mean)
    rp, ci = torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col_ind).cuda()
    M = b.cmrs_from_csr(rp, ci, torch.from_numpy(a.val).cuda(), a.cols, h, dtype=dtype)
    x = inputs.uniform_vector(a.cols, 5)
    x = x if dtype == 0 else x.astype(np.float32)
    xd = torch.from_numpy(x).cuda()
    y = b.cmrs_spmv(M, xd, torch.full((a.rows,), float("nan"), dtype=xd.dtype, device="cuda"), b.CMRS_VARIANT_MERGE)
    b.cmrs_spmv_check(M, b.CMRS_VARIANT_MERGE)
    vq = a.val if dtype == 0 else orc.decode(orc.encode(a.val, dtype), dtype, a.nnz)
    yref, absy = orc.csr_spmv(a.row_ptr, a.col_ind, vq, x.astype(np.float64))
    # FP64: the library's bar; FP32 accumulation: any order of n exact products
    tol = 1e-12 * absy if dtype == 0 else (np.diff(a.row_ptr) + 2) * 2.0**-24 * absy
    assert (np.abs(y.cpu().numpy().astype(np.float64) - yref) <= tol).all()
    assert torch.equal(y, b.cmrs_spmv(M, xd, variant=b.CMRS_VARIANT_MERGE))
