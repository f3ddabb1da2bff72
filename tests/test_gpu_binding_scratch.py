"""Scratch memory the binding does not zero: every entry point that gets it clears its own status word."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1203_2946_gb300 import build
    build.build()
    from paper_1203_2946_gb300 import binding
    return binding


def test_status_words_of_unzeroed_scratch(b, monkeypatch):
    blocks = []

    def ones(nbytes, device):
        blocks.append(torch.full((max(int(nbytes), 256),), 255, dtype=torch.uint8, device=device))
        return blocks[-1]

    monkeypatch.setattr(b, "_scratch", ones)
    rp = torch.tensor([0, 2, 2, 5], dtype=torch.int32, device="cuda")
    ci = torch.tensor([0, 2, 0, 1, 2], dtype=torch.int32, device="cuda")
    va = torch.arange(5, dtype=torch.float64, device="cuda")
    for flags in (0, b.CMRS_SORTED):
        A = b.cmrs_from_csr(rp, ci, va, 3, 32, flags=flags)
        out = b.cmrs_to_csr(A)
        assert [t.tolist() for t in out[:2]] == [rp.tolist(), ci.tolist()]
        assert out[2].view(torch.float64)[:5].tolist() == va.tolist()
        assert b.cmrs_to_csr(A, with_values=False)[2] is None
    b.cmrs_pad(b.cmrs_from_csr(rp, ci, va, 3, 32), 1)
    assert blocks and all(int(t[:4].view(torch.int32)) == 0 for t in blocks)
