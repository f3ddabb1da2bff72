"""The stream a call without a stream argument runs on: the caller's current one, on the caller's current device."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def b():
    from paper_1203_2946_gb300 import build
    build.build()
    from paper_1203_2946_gb300 import binding
    return binding


def test_current_stream_handle(b):
    torch.zeros(1, device="cuda")
    assert b._stream(None) == torch.cuda.current_stream().cuda_stream
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        assert b._stream(None) == s.cuda_stream != torch.cuda.default_stream().cuda_stream
    assert b._stream(s) == s.cuda_stream
    assert b._stream(s.cuda_stream) == s.cuda_stream


def test_workspaces_that_are_not_zeroed(b):
    """Conversions and features on scratch memory full of ones: the entry points clear what they read."""
    rp = torch.tensor([0, 2, 2, 5], dtype=torch.int32, device="cuda")
    ci = torch.tensor([0, 2, 0, 1, 2], dtype=torch.int32, device="cuda")
    va = torch.arange(5, dtype=torch.float64, device="cuda")
    want = None
    for fill in (0, 255):
        blocks = [torch.full((1 << 20,), fill, dtype=torch.uint8, device="cuda") for _ in range(8)]
        del blocks  # back to torch's pool: the next small allocations reuse it
        got = []
        for flags in (0, b.CMRS_SORTED):
            A = b.cmrs_from_csr(rp, ci, va, 3, 32, flags=flags)
            got += [A.strip_ptr.tolist(), A.col_packed[:5].tolist(), b.stored_values(A).tolist()]
            got += [t[:5].tolist() for t in b.cmrs_to_csr(A)[:2]]
        P = b.cmrs_pad(b.cmrs_from_csr(rp, ci, va, 3, 32), 1)
        got += [P.strip_ptr.tolist(), P.col_packed.tolist(), b.cmrs_features(rp, ci).tolist()]
        assert want is None or got == want
        want = got
