"""cmrs_pad_fill where its passes change form: full passes (each copied while the next is planned) next to general ones
and runs of passes alike, strips past the stage, and the plan-free layout at height x M = 32.  The arrangement equals the
oracle's bit for bit."""
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


LENGTHS = {
    "mixed": lambda r: r.integers(4, 61, 3001),                              # mostly full passes
    "equal": lambda r: np.full(1000, 24),                                    # the last pass alone is general
    "two_levels": lambda r: np.where(np.arange(2001) % 3 == 0, 40, 7),       # full, then alike
    "long_rows": lambda r: np.where(np.arange(700) % 97 == 5, 1500, r.integers(0, 6, 700)),  # past the stage, one row
    "some_left": lambda r: np.where(np.arange(640) % 32 < 17, 65, 1),        # 17 rows of 32: one more than M = 2 takes
}


@pytest.mark.parametrize("h,slots", [(32, 1), (16, 2), (8, 4), (4, 8), (32, 2), (32, 4), (16, 8), (9, 4)])
@pytest.mark.parametrize("case", sorted(LENGTHS))
@pytest.mark.parametrize("dtype", [0, 3])
def test_passes_of_each_form(b, case, h, slots, dtype):
    L = LENGTHS[case](np.random.default_rng(h + slots))
    a = inputs.from_lengths(L, 30000, seed=7)
    M = b.cmrs_from_csr(torch.from_numpy(a.row_ptr).cuda(), torch.from_numpy(a.col_ind).cuda(),
                        torch.from_numpy(a.val).cuda(), a.cols, h, dtype=dtype)
    P = b.cmrs_pad(M, slots)
    ref = orc.pad_arrange(a.rows, h, M.strip_ptr.cpu().numpy(), M.col_packed.cpu().numpy()[:M.nnz].view(np.uint32), slots)
    assert np.array_equal(P.strip_ptr.cpu().numpy(), ref["strip_ptr"])
    assert np.array_equal(P.col_packed.cpu().numpy()[:P.nnz].view(np.uint32), ref["packed"])
    v0, v1, src = b.stored_values(M).cpu().numpy(), b.stored_values(P).cpu().numpy(), ref["src"]
    for part in range(2 if dtype == 3 else 1):
        want = np.zeros_like(v1[:P.nnz])
        want[src >= 0] = v0[part * M.nnz:(part + 1) * M.nnz][src[src >= 0]]
        assert np.array_equal(v1[part * P.nnz:(part + 1) * P.nnz].view(np.uint8), want.view(np.uint8))
