"""Column-sorted conversion of invalid CRS input: refused with an error code,
nothing written outside the given arrays."""
import ctypes

import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu

GUARD = 1 << 20  # bytes either side of an array


@pytest.fixture(scope="module")
def b():
    from paper_1203_2946_gb300 import build
    build.build()
    from paper_1203_2946_gb300 import binding
    return binding


class Guarded:
    """An array of nbytes with guard bytes on both sides of it."""

    def __init__(self, nbytes):
        self.n = nbytes
        self.whole = torch.full((GUARD + (nbytes + 255) // 256 * 256 + GUARD,), 0xA5, dtype=torch.uint8, device="cuda")

    def ptr(self):
        return self.whole.data_ptr() + GUARD

    def intact(self):
        return bool((self.whole[:GUARD] == 0xA5).all() and (self.whole[GUARD + self.n:] == 0xA5).all())


def convert_sorted(b, row_ptr, nnz, cols, height):
    """Status of cmrs_from_csr with CMRS_SORTED, and whether every array's guards survived."""
    rows = row_ptr.size - 1
    rp = torch.from_numpy(row_ptr.astype(np.int32)).cuda()
    ci = torch.arange(nnz, dtype=torch.int32, device="cuda") % cols
    va = torch.ones(nnz, dtype=torch.float64, device="cuda")
    n = ctypes.c_size_t()
    assert b.lib().cmrs_from_csr_workspace(rows, nnz, height, b.CMRS_SORTED, b.CMRS_F64, ctypes.byref(n)) == 0
    sp, pk, vo, ws = Guarded(4 * (-(-rows // height) + 1)), Guarded(4 * nnz), Guarded(8 * nnz), Guarded(n.value)
    out = b.cmrs_matrix()
    rc = b.lib().cmrs_from_csr(rows, cols, nnz, rp.data_ptr(), ci.data_ptr(), va.data_ptr(), b.CMRS_F64, height,
                               b.CMRS_SORTED, b.CMRS_F64, sp.ptr(), pk.ptr(), vo.ptr(), ws.ptr(), n.value,
                               torch.cuda.current_stream().cuda_stream, ctypes.byref(out))
    torch.cuda.synchronize()
    return rc, all(g.intact() for g in (sp, pk, vo, ws))


# every other strip valid by itself and holding all nnz entries: for a warp, the CTA list, the radix list
@pytest.mark.parametrize("nnz", [200, 300, 1025, 6144, 7000, 20_000])
@pytest.mark.parametrize("height,strips", [(1, 20_001), (2, 10_001), (32, 1001)])
def test_overlapping_strips(b, nnz, height, strips):
    rp = np.empty(strips * height + 1, np.int64)
    s = np.arange(strips * height) // height
    rp[:-1] = np.where(s % 2 == 0, 0, nnz)
    rp[-1] = nnz
    assert convert_sorted(b, rp, nnz, 5000, height) == (4, True)


# no strip to sort: entries without rows are an invalid RowPtr, not a launch of no blocks
@pytest.mark.parametrize("first", [0, 1])
@pytest.mark.parametrize("nnz", [1, 300, 7000])
def test_entries_without_rows(b, nnz, first):
    assert convert_sorted(b, np.array([first * nnz]), nnz, 5000, 4) == (4, True)
