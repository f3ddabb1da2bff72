"""Conversions of matrices whose strips are all longer than a warp's stage, bit for bit against the oracle."""
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


LENGTHS = {32: lambda r: r.integers(100, 260, 150), 16: lambda r: r.integers(200, 500, 70), 8: lambda r: r.integers(400, 700, 41)}


def matrix(h):
    return inputs.from_lengths(LENGTHS[h](np.random.default_rng(h)), 9000, seed=7)


def convert(b, a, h, dtype, flags=0):
    return b.cmrs_from_csr(torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col_ind).cuda(),
                           torch.from_numpy(a.val).cuda(), a.cols, h, flags=flags, dtype=dtype)


@pytest.mark.parametrize("h,slots", [(32, 1), (32, 2), (16, 2), (16, 8), (8, 4), (8, 8)])
@pytest.mark.parametrize("dtype", [0, 1, 2, 3])
def test_pad(b, h, slots, dtype):
    M = convert(b, matrix(h), h, dtype)
    P = b.cmrs_pad(M, slots)
    ref = orc.pad_arrange(M.rows, h, M.strip_ptr.cpu().numpy(), M.col_packed.cpu().numpy()[:M.nnz].view(np.uint32), slots)
    assert np.array_equal(P.strip_ptr.cpu().numpy(), ref["strip_ptr"])
    assert np.array_equal(P.col_packed.cpu().numpy()[:P.nnz].view(np.uint32), ref["packed"])
    src = torch.from_numpy(ref["src"].astype(np.int64)).cuda()
    v0, v1 = b.stored_values(M), b.stored_values(P)
    for k in range(2 if dtype == 3 else 1):
        want = torch.where(src >= 0, v0[k * M.nnz:(k + 1) * M.nnz][src.clamp(min=0)], 0)
        assert torch.equal(v1[k * P.nnz:(k + 1) * P.nnz], want)


# sorted strips to CRS: walked (short, long, few rows, one strip far past the stage) and staged
TO_CSR = {"short": (lambda r: r.integers(0, 9, 700), 4), "staged": (lambda r: r.integers(20, 60, 700), 8),
          "staged_tall": (lambda r: r.integers(4, 9, 900), 32), "long": (lambda r: r.integers(100, 300, 300), 16),
          "one_row": (lambda r: r.integers(600, 900, 40), 1), "one_long": (lambda r: np.where(np.arange(800) == 300, 8000, 30), 8)}


@pytest.mark.parametrize("case", sorted(TO_CSR))
@pytest.mark.parametrize("dtype", [0, 1, 2, 3])
def test_sorted_to_csr(b, case, dtype):
    make, h = TO_CSR[case]
    a = inputs.from_lengths(make(np.random.default_rng(2)), 9000, seed=3)
    M, plain = convert(b, a, h, dtype, b.CMRS_SORTED), convert(b, a, h, dtype)
    rp, ci, v = b.cmrs_to_csr(M)
    assert np.array_equal(rp.cpu().numpy(), a.row_ptr) and np.array_equal(ci.cpu().numpy(), a.col_ind)
    width = {0: 8, 1: 4, 2: 2, 3: 2}[dtype]
    pad = b.lib().cmrs_pad8(a.nnz) * 2
    for at in (0, pad) if dtype == 3 else (0,):  # columns were in order: the plain matrix's values, byte for byte
        assert torch.equal(v[at:at + width * a.nnz], plain.val[at:at + width * a.nnz])
