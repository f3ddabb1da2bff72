"""CRS -> CMRS at the sizes and values where the conversion kernels' paths
change, bit for bit: FP32 sources against the same values given as doubles,
row groups with and without empty rows."""
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


def dev(a):
    return torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col_ind).cuda()


@pytest.mark.parametrize("dtype", [1, 2, 3])
def test_float_source_equals_double_source(b, dtype):
    rng = np.random.default_rng(2)
    bits = np.concatenate([rng.integers(0, 2**32, 5000, dtype=np.uint64).astype(np.uint32),  # any pattern, NaNs among them
                           np.array([0x7f800001, 0xff812345, 0x7fffffff, 0x7f800000, 0xff800000, 0, 0x80000000, 1,
                                     0x007fffff, 0x00800000, 0x7f7fffff, 0x3f7fffff, 0x3f808000, 0x3f818000],
                                    np.uint32)])
    n = bits.size
    v32 = torch.from_numpy(bits.view(np.float32)).cuda()
    rp = torch.arange(n + 1, dtype=torch.int32, device="cuda")
    ci = torch.arange(n, dtype=torch.int32, device="cuda")
    with np.errstate(invalid="ignore"):
        v64 = torch.from_numpy(bits.view(np.float32).astype(np.float64)).cuda()
    got = b.stored_values(b.cmrs_from_csr(rp, ci, v32, n, 8, dtype=dtype))
    want = b.stored_values(b.cmrs_from_csr(rp, ci, v64, n, 8, dtype=dtype))
    w = torch.int32 if dtype == 1 else torch.int16
    assert torch.equal(got.view(w), want.view(w))


@pytest.mark.parametrize("h", [1, 5, 32])
@pytest.mark.parametrize("lengths", ["no_empty", "some_empty", "batch_edges", "tail"])
def test_row_of_each_entry(b, h, lengths):
    rng = np.random.default_rng(h)
    L = {"no_empty": rng.integers(1, 40, 1000),
         "some_empty": rng.integers(0, 3, 1000),
         "batch_edges": np.tile([32, 31, 1, 64, 128, 96, 33, 127], 50),  # rows that end where a batch of 32 does
         "tail": np.concatenate([rng.integers(1, 9, 96), [700]])}[lengths]
    a = inputs.from_lengths(L, 5000, seed=8)
    rp, ci = dev(a)
    M = b.cmrs_from_csr(rp, ci, torch.from_numpy(a.val).cuda(), a.cols, h)
    ref = orc.csr_to_cmrs(a.row_ptr, a.col_ind, a.val, a.cols, h)
    assert np.array_equal(M.strip_ptr.cpu().numpy(), ref["strip_ptr"])
    assert np.array_equal(M.col_packed.cpu().numpy()[:a.nnz].view(np.uint32), ref["packed"])
    assert np.array_equal(b.stored_values(M).cpu().numpy(), ref["val"])
    assert M.struct.max_strip_nnz == np.diff(ref["strip_ptr"]).max()
