"""The selector's kernels at the sizes where their paths change: features of
row groups either side of the shared-memory stage and of the short-row bound
(and of a column array no bulk copy can read), the network at sizes that fit a
block's shared memory and at sizes that do not."""
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
    rng = np.random.default_rng(4)
    if kind == "short":  # every group staged; empty rows and groups; a last group of 5 rows
        L = rng.integers(0, 12, 32 * 40 + 5)
        L[64:128] = 0
        return L
    if kind == "stage_edge":  # mean 64: stage of 2,048; groups of exactly 2,048 and 2,049 entries, rows of 63..65
        L = np.full(32 * 30 + 1, 64)
        L[32] += 1
        L[64], L[65] = 63, 65
        return L
    if kind == "long":  # groups read from global memory: short and long rows side by side
        L = rng.integers(0, 5, 32 * 20 + 17)
        L[[3, 100, 101, 500, 656]] = [9000, 65, 64, 8192, 511]
        return L
    return np.array([0, 0, 3])


@pytest.mark.parametrize("kind", ["short", "stage_edge", "long", "tiny"])
@pytest.mark.parametrize("offset", [0, 1])
def test_features_either_side_of_the_stage(b, kind, offset):
    a = inputs.from_lengths(lengths(kind), 20000, seed=6)
    rp = torch.from_numpy(a.row_ptr).cuda()
    buf = torch.zeros(a.nnz + 8, dtype=torch.int32, device="cuda")
    ci = buf[offset:offset + a.nnz]  # offset 1: 4 bytes past a 16-byte boundary
    ci.copy_(torch.from_numpy(a.col_ind))
    f = b.cmrs_features(rp, ci).cpu().numpy()
    # integer sums and the oracle's operations in its order: log2 alone may differ, by an ulp or two
    assert np.allclose(f, orc.features(a.row_ptr, a.col_ind), rtol=1e-14, atol=1e-14)


@pytest.mark.parametrize("B,nin,nh,nout", [(1, 32, 64, 21), (3, 5, 7, 2), (6, 31, 33, 32), (257, 32, 64, 21),
                                           (9, 24, 140, 18), (5, 300, 200, 33)])
def test_network_sizes(b, B, nin, nh, nout):
    """Blocks of four samples (whole and partial), layers either side of a
    warp, networks too large for a block (140 and 200 hidden units).  Each
    result is a chain of at most nin + 2 nh + nout + B FP32 roundings of sums
    of its own magnitude, so its error is below (that count) 2^-24 in the
    2-norm with room for the layers' growth: 16 times that."""
    rng = np.random.default_rng(B + nh)
    shapes = [(nh, nin), (nh,), (nh, nh), (nh,), (nout, nh), (nout,)]
    p32 = [(rng.normal(0, 1 / np.sqrt(s[-1]), s)).astype(np.float32) for s in shapes]
    X, T = rng.normal(0, 1, (B, nin)).astype(np.float32), rng.normal(0, 1, (B, nout)).astype(np.float32)
    P = torch.from_numpy(np.concatenate([p.ravel() for p in p32])).cuda()
    Xd, Td = torch.from_numpy(X).cuda(), torch.from_numpy(T).cuda()
    acts = b.cmrs_mlp_forward(Xd, P, nh, nout)
    grads, loss = b.cmrs_mlp_backward(Xd, Td, P, acts, nh, nout)
    ref_loss, g, fw = orc.mlp_loss_grad(X.astype(np.float64), T.astype(np.float64),
                                        *[p.astype(np.float64) for p in p32])
    tol = 16 * (nin + 2 * nh + nout + B) * 2.0**-24

    def close(got, ref):
        ref = np.asarray(ref, np.float64).ravel()
        assert np.linalg.norm(got.astype(np.float64).ravel() - ref) <= tol * np.linalg.norm(ref)

    a = acts.cpu().numpy()
    for k, name in enumerate(("Z1", "H1", "Z2", "H2")):
        close(a[k * B * nh:(k + 1) * B * nh], fw[name])
    close(a[4 * B * nh:4 * B * nh + B * nout], fw["O"])
    close(loss.cpu().numpy(), [ref_loss])
    at = 0
    for name in ("W1", "b1", "W2", "b2", "W3", "b3"):
        n = g[name].size
        close(grads[at:at + n].cpu().numpy(), g[name])
        at += n
