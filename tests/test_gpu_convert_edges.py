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


def csr(lengths, cols, seed, order="ordered"):
    """Rows of the given lengths; columns increasing, or shuffled inside each row, or drawn with repeats (equal columns
    in one row), shuffled or ordered."""
    a = inputs.from_lengths(lengths, cols, seed=seed)
    if order == "ordered":
        return a
    rng = np.random.default_rng(seed)
    ci = a.col_ind.copy()
    for r in range(a.rows):
        p, q = a.row_ptr[r], a.row_ptr[r + 1]
        ci[p:q] = rng.permutation(ci[p:q]) if order == "shuffled" else rng.integers(0, min(50, cols), q - p)
        if order == "ordered_repeats":
            ci[p:q].sort()
    return inputs.CSR(a.rows, a.cols, a.row_ptr, ci, a.val, a.name)


SORT_CASES = {
    "short": (lambda rng: rng.integers(0, 12, 501), 4000),  # warp strips, empty rows, a last strip cut short
    "equal_columns": (lambda rng: np.full(320, 7), 9),      # nearly every column in every row: ties across rows
    "full_rows": (lambda rng: np.full(96, 32), 32),         # dense strips: as many ties as rows
    # a warp's buffer, a CTA's, the radix sort: strips either side of each bound at some height below
    "bounds": (lambda rng: np.concatenate([np.full(64, 8), [256 - 8 * 7, 257, 1024, 1025, 6144, 6145, 9000], np.full(57, 8)]),
               20000),
    "long_mean": (lambda rng: rng.integers(100, 300, 160), 3000),  # CTA strips throughout at height 32
}


@pytest.mark.parametrize("h", [1, 2, 3, 6, 8, 16, 32])
@pytest.mark.parametrize("case", sorted(SORT_CASES))
@pytest.mark.parametrize("order", ["ordered", "shuffled", "repeats", "ordered_repeats"])
def test_sorted_strips(b, case, h, order):
    make, cols = SORT_CASES[case]
    a = csr(make(np.random.default_rng(3)), cols, 5, order)
    rp, ci = dev(a)
    M = b.cmrs_from_csr(rp, ci, torch.from_numpy(a.val).cuda(), a.cols, h, flags=b.CMRS_SORTED)
    ref = orc.csr_to_cmrs(a.row_ptr, a.col_ind, a.val, a.cols, h, sorted_=True)
    assert np.array_equal(M.strip_ptr.cpu().numpy(), ref["strip_ptr"])
    assert np.array_equal(M.col_packed.cpu().numpy()[:a.nnz].view(np.uint32), ref["packed"])
    assert np.array_equal(b.stored_values(M).cpu().numpy(), ref["val"])
    assert M.struct.max_strip_nnz == np.diff(ref["strip_ptr"]).max()
    rp2, ci2, v2 = b.cmrs_to_csr(M)
    r3 = orc.cmrs_to_csr(a.rows, h, ref["strip_ptr"], ref["packed"], ref["val"])
    assert np.array_equal(rp2.cpu().numpy(), r3["row_ptr"])
    assert np.array_equal(ci2.cpu().numpy(), r3["col_ind"])
    assert np.array_equal(v2.view(torch.float64).cpu().numpy()[:a.nnz], r3["val"])


@pytest.mark.parametrize("src", [torch.float32, torch.float64])
@pytest.mark.parametrize("dtype", [0, 1, 2, 3])
def test_sorted_values_every_form(b, dtype, src):
    a = csr(np.random.default_rng(1).integers(0, 90, 300), 900, 2)
    rp, ci = dev(a)
    va = torch.from_numpy(a.val).cuda().to(src)
    plain = b.cmrs_from_csr(rp, ci, va, a.cols, 12, dtype=dtype)
    M = b.cmrs_from_csr(rp, ci, va, a.cols, 12, flags=b.CMRS_SORTED, dtype=dtype)
    order = torch.from_numpy(orc.csr_to_cmrs(a.row_ptr, a.col_ind, a.val, a.cols, 12, sorted_=True)["src"].astype(np.int64)).cuda()
    v, w = b.stored_values(plain), b.stored_values(M)
    for k in range(2 if dtype == 3 else 1):
        assert torch.equal(v[k * a.nnz:(k + 1) * a.nnz][order], w[k * a.nnz:(k + 1) * a.nnz])


@pytest.mark.parametrize("what", ["column", "negative", "row_ptr", "last"])
def test_sorted_invalid_input_is_refused(b, what):
    a = csr(np.random.default_rng(1).integers(1, 90, 3000), 900, 2)
    rp, ci = a.row_ptr.copy(), a.col_ind.copy()
    if what == "column":
        ci[1234] = 900
    elif what == "negative":
        ci[5] = -1
    elif what == "row_ptr":
        rp[700] = rp[702]
    else:
        rp[-1] -= 1
    with pytest.raises(b.CmrsError) as e:
        b.cmrs_from_csr(torch.from_numpy(rp).cuda(), torch.from_numpy(ci).cuda(), torch.from_numpy(a.val).cuda(), 900, 8,
                        flags=b.CMRS_SORTED)
    assert e.value.code == 4


@pytest.mark.parametrize("length", [257, 1024, 1025, 6144, 6145])
def test_sorted_out_of_order_strips_fill_the_lists(b, length):
    # equal strips, every one out of order: as many listed strips as nnz has room for
    h, n = 4, 24
    kr = np.tile([length - 3 * (length // 4)] + 3 * [length // 4], n)
    a = csr(kr, 9000, 7, "shuffled")
    rp, ci = dev(a)
    M = b.cmrs_from_csr(rp, ci, torch.from_numpy(a.val).cuda(), a.cols, h, flags=b.CMRS_SORTED)
    ref = orc.csr_to_cmrs(a.row_ptr, a.col_ind, a.val, a.cols, h, sorted_=True)
    assert np.array_equal(M.col_packed.cpu().numpy()[:a.nnz].view(np.uint32), ref["packed"])
    assert np.array_equal(b.stored_values(M).cpu().numpy(), ref["val"])
