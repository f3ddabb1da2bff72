"""What a user of this library has it do, as cases that can be timed.

A case is a dict of plain values; prepare(case, seed) makes on the GPU what a
program has in hand before the call (the CRS matrix, or the CMRS matrix it
keeps, x, the network), run(state) is one pass through the public entry points
of paper_1203_2946_gb300.binding, work(case) the bytes and operations the pass
cannot do without, exact(case, seed) its result in 64 bits from plain torch.

Kinds of case:
  spmv     y = A x with the default variant, on plain, padded (Section 6.6) or
           column-sorted (Section 4) strips
  spmm     many uneven matrices with k right-hand sides each, one launch
  pad      CRS -> CMRS -> padded CMRS (what a program pays once per matrix)
  sort     CRS -> column-sorted CMRS, and back to CRS
  setup    a new matrix: choose its form with the trained selector, convert
           it, multiply once
  train    one training step of the selector's network (forward, backward,
           Adam)

Matrices come from the families and sizes the benchmark and the selector
corpus use.  The random ones draw one uniform column in each of the L equal
strata of a row's column range, which keeps columns distinct and increasing.
"""
from __future__ import annotations

import math
import os

import torch

from paper_1203_2946_gb300 import binding as b
from paper_1203_2946_gb300 import selector

VALUE_BYTES = {"f64": 8, "f32": 4, "bf16": 2, "bf16x2": 4}
CARD = "cuda"


def listed():
    return [
        # an iteration of a solver on a small grid: one short launch, its latency and the call itself
        dict(name="spmv_lap2d_64_f64", kind="spmv", family="lap2d", n=64 * 64, form="plain", height=4, slots=0,
             dtype="f64"),
        # the 3-D stencil a solver multiplies thousands of times, as converted (no padding), FP64
        dict(name="spmv_st27_128_f64_plain", kind="spmv", family="stencil27", n=128**3, form="plain", height=4,
             slots=0, dtype="f64"),
        # the same in the modified form a program keeps for the fastest FP64 product
        dict(name="spmv_st27_128_f64_padded", kind="spmv", family="stencil27", n=128**3, form="padded", height=32,
             slots=1, dtype="f64"),
        # the same with values as BF16 pairs, for the inner products of a mixed-precision solver
        dict(name="spmv_st27_128_bf16x2_padded", kind="spmv", family="stencil27", n=128**3, form="padded", height=32,
             slots=1, dtype="bf16x2"),
        # a graph: power-law row lengths, random columns, FP32 (a PageRank-like iteration)
        dict(name="spmv_powerlaw_4m_f32", kind="spmv", family="powerlaw", n=4_194_304, alpha=2.1, kmax=100_000,
             form="plain", height=32, slots=0, dtype="f32"),
        # an unstructured mesh: rows of 4..60 entries in a band, FP64, two slots per row
        dict(name="spmv_irregular_2m_f64_padded", kind="spmv", family="banded", n=2_097_152, width=2048, lo=4, hi=60,
             form="padded", height=32, slots=2, dtype="f64"),
        # the paper's own kernel and layout: column-sorted strips of 4 rows, FP64
        dict(name="spmv_st27_128_f64_sorted", kind="spmv", family="stencil27", n=128**3, form="sorted", height=4,
             slots=0, dtype="f64"),
        # many systems at once: 64 banded matrices of 1,000 to 200,000 rows, k of 1, 4, 8 or 32 each
        dict(name="spmm_batch_64", kind="spmm", batch=64, n_lo=1000, n_hi=200_000, k="1,4,8,32", height=1),
        # conversion of an irregular matrix to the padded form, FP32
        dict(name="pad_irregular_2m_f32", kind="pad", family="banded", n=2_097_152, width=2048, lo=4, hi=60,
             height=32, slots=2, dtype="f32"),
        # conversion to column-sorted strips and back, at a size that divides into nothing
        dict(name="sort_uniform_1m_f64", kind="sort", family="uniform", n=1_000_003, mu=20.0, height=16, dtype="f64"),
        # a matrix never seen before: select, convert, first product
        dict(name="setup_banded_400k_f32", kind="setup", family="banded", n=400_009, width=1024, lo=20, hi=60,
             dtype="f32"),
        # a training step of the selector's network on its usual batch
        dict(name="train_256", kind="train", batch=256, nh=64),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _draw_matrix(rng, most=60e6):
    """A family and size of the selector corpus' range, at most `most` entries."""
    fam = rng.choice(["lap2d", "stencil27", "stencil7", "banded", "banded", "blockdiag", "powerlaw", "uniform"])
    n = _log(rng, 4000, 4.2e6)
    c = dict(family=fam, n=n)
    if fam == "banded":
        lo = _log(rng, 2, 100)
        c.update(lo=lo, hi=min(200, max(lo + 1, int(lo * rng.uniform(1.2, 8.0)))), width=rng.randint(256, 2048))
    elif fam == "blockdiag":
        c["block"] = rng.randint(4, 32)
    elif fam == "powerlaw":
        c.update(alpha=round(rng.uniform(1.9, 2.6), 2), kmax=max(64, min(100_000, n // 4)))
    elif fam == "uniform":
        c["mu"] = round(math.exp(rng.uniform(math.log(2.0), math.log(200.0))), 1)
    while _nnz(c) > most:
        c["n"] = int(c["n"] * 0.6)
        if fam == "powerlaw":
            c["kmax"] = max(64, min(c["kmax"], c["n"] // 4))
    return c


def draw(rng):
    kind = rng.choice(["spmv"] * 5 + ["spmm", "pad", "sort", "setup", "train"])
    if kind == "train":
        return dict(kind="train", batch=_log(rng, 16, 2000), nh=rng.choice([16, 32, 48, 64]))
    if kind == "spmm":
        hi = _log(rng, 5000, 200_000)
        return dict(kind="spmm", batch=rng.randint(2, 64), n_lo=1000, n_hi=hi, height=rng.choice([1, 1, 1, 2, 4]),
                    k=rng.choice(["1,4,8,32", "1,4,8,32", "1,2,3,5", "4,8,16", "1", "32"]))
    c = dict(kind=kind, **_draw_matrix(rng, 60e6 if kind == "spmv" else 30e6))
    if kind == "setup":
        return dict(c, dtype="f32")
    c["dtype"] = rng.choice(["f64", "f64", "f32", "f32", "bf16", "bf16x2"])
    if c["family"] == "powerlaw" and kind != "spmv":
        c["kmax"] = min(c["kmax"], 2000)
    if kind == "sort":
        return dict(c, height=rng.choice([2, 4, 6, 8, 12, 16, 32]))
    form = "padded" if kind == "pad" else rng.choice(["plain", "plain", "padded", "sorted"])
    if form == "padded":  # the three forms the selector chooses between
        h, m = rng.choice([(32, 1), (32, 2), (16, 8)]) if c["family"] != "powerlaw" else (16, 8)
    else:
        h, m = rng.choice([1, 2, 4, 4, 6, 8, 12, 16, 32]), 0
    if c["family"] == "powerlaw" and form != "plain":
        c["kmax"] = min(c["kmax"], 2000)
    c.update(height=h, slots=m)
    return c if kind == "pad" else dict(c, form=form)


# ------------------------------------------------------------------ matrices (CRS, on the GPU)
def _gen(seed):
    g = torch.Generator(device=CARD)
    g.manual_seed(int(seed) * 1000003 + 17)
    return g


def _edge(case):
    d = 2 if case["family"] == "lap2d" else 3
    return max(3, int(round(case["n"] ** (1.0 / d))))


def _rows(case):
    if case["family"] == "lap2d":
        return _edge(case) ** 2
    if case["family"] in ("stencil27", "stencil7"):
        return _edge(case) ** 3
    return case["n"]


def _zipf_table(alpha, kmax):
    k = torch.arange(1, kmax + 1, device=CARD, dtype=torch.float64)
    p = k.pow(-alpha)
    tail = (kmax + 0.5) ** (1.0 - alpha) / (alpha - 1.0)  # lengths past kmax are clipped to it
    p[-1] += tail
    return p / p.sum()


def _nnz(case):
    """Entries of the matrix: exact for the grids, the mean for the random families."""
    f, n = case["family"], case["n"]
    if f == "lap2d":
        m = _edge(case)
        return 5 * m * m - 4 * m
    if f == "stencil27":
        return (3 * _edge(case) - 2) ** 3
    if f == "stencil7":
        m = _edge(case)
        return 7 * m**3 - 6 * m * m
    if f == "banded":
        return int(n * (case["lo"] + case["hi"]) / 2)
    if f == "blockdiag":
        q, r = divmod(n, case["block"])
        return q * case["block"] ** 2 + r * r
    if f == "uniform":
        return int(n * case["mu"])
    a, m = case["alpha"], case["kmax"]
    num = den = 0.0
    for k in range(1, m + 1):
        num += k ** (1.0 - a)
        den += k**-a
    tail = (m + 0.5) ** (1.0 - a) / (a - 1.0)
    return int(n * (num + m * tail) / (den + tail))


def _grid(case, g, dtype):
    """A stencil on a cube or square, natural order, neighbours outside it dropped."""
    m = _edge(case)
    d = 2 if case["family"] == "lap2d" else 3
    offs = [()]
    for _ in range(d):
        offs = [o + (s,) for o in offs for s in (-1, 0, 1)]
    if case["family"] in ("lap2d", "stencil7"):
        offs = [o for o in offs if sum(abs(s) for s in o) <= 1]
    n = m**d
    idx = torch.arange(n, device=CARD, dtype=torch.int64)
    at = [(idx // m ** (d - 1 - i)) % m for i in range(d)]
    valid = torch.ones((n, len(offs)), dtype=torch.bool, device=CARD)
    for k, o in enumerate(offs):
        for i, s in enumerate(o):
            if s:
                valid[:, k] &= (at[i] + s >= 0) & (at[i] + s < m)
    step = torch.tensor([sum(s * m ** (d - 1 - i) for i, s in enumerate(o)) for o in offs], device=CARD)
    full = torch.rand((n, len(offs)), generator=g, device=CARD, dtype=dtype) * 2 - 1
    mid = offs.index((0,) * d)
    if case["family"] == "lap2d":
        full.fill_(-1.0)
        full[:, mid] = 4.0
    else:  # strictly diagonally dominant
        full[:, mid] = 0.0
        full[:, mid] = (full.abs() * valid).sum(1) + 1.0
    return n, valid.sum(1), (idx[:, None] + step[None, :])[valid], full[valid]


def _crs(case, seed, dtype):
    """(rows, row_ptr, col_ind, val): int32 indices, columns increasing in each row.  Row lengths belong to the case
    (as a mesh's or a graph's do, and so that the outputs of a conversion keep their sizes), columns and values to the
    seed."""
    g, gl = _gen(seed), _gen(3)
    f, n = case["family"], case["n"]
    if f in ("lap2d", "stencil27", "stencil7"):
        n, lengths, col, val = _grid(case, g, dtype)
    else:
        i = torch.arange(n, device=CARD, dtype=torch.int64)
        lo, width = torch.zeros_like(i), torch.full_like(i, n)
        if f == "banded":
            w = min(case["width"], n)
            lengths = torch.randint(min(case["lo"], w), min(case["hi"], w) + 1, (n,), generator=gl, device=CARD)
            lo, width = (i - w // 2).clamp(0, n - w), torch.full_like(i, w)
        elif f == "blockdiag":
            lo = i // case["block"] * case["block"]
            lengths = width = (lo + case["block"]).clamp(max=n) - lo
        elif f == "powerlaw":
            cdf = _zipf_table(case["alpha"], case["kmax"]).cumsum(0)
            u = torch.rand(n, generator=gl, device=CARD, dtype=torch.float64)
            lengths = (torch.searchsorted(cdf, u) + 1).clamp(max=case["kmax"])
        else:  # uniform: Poisson lengths, some rows empty where mu is small
            mu = torch.full((n,), case["mu"], device=CARD, dtype=torch.float32)
            lengths = torch.poisson(mu, generator=gl).to(torch.int64).clamp(max=n)
        row = torch.repeat_interleave(i, lengths)
        j = torch.arange(row.numel(), device=CARD, dtype=torch.int64) - (lengths.cumsum(0) - lengths)[row]
        L, w = lengths[row], width[row]
        b0, b1 = j * w // L, (j + 1) * w // L
        u = torch.rand(row.numel(), generator=g, device=CARD, dtype=torch.float64)
        col = lo[row] + b0 + torch.minimum((u * (b1 - b0)).to(torch.int64), b1 - b0 - 1)
        val = torch.randn(row.numel(), generator=g, device=CARD, dtype=dtype)
    rp = torch.zeros(n + 1, dtype=torch.int64, device=CARD)
    torch.cumsum(lengths, 0, out=rp[1:])
    return n, rp.to(torch.int32), col.to(torch.int32), val


def _vector(n, seed, dtype):
    return torch.rand(n, generator=_gen(seed + 77777), device=CARD, dtype=dtype) * 2 - 1


def _input_type(case):
    return torch.float64 if case["dtype"] == "f64" else torch.float32


# ------------------------------------------------------------------ the batch
def _batch(case):
    """(rows, band width, right-hand sides) of each matrix, fixed by the case."""
    sizes = torch.Generator().manual_seed(7)
    ks = [int(k) for k in case["k"].split(",")]
    specs = []
    for _ in range(case["batch"]):
        n = int(torch.randint(case["n_lo"], case["n_hi"] + 1, (1,), generator=sizes))
        w = int(torch.randint(64, 2049, (1,), generator=sizes))
        specs.append((n, w, ks[int(torch.randint(0, len(ks), (1,), generator=sizes))]))
    return specs


def _batch_data(case, seed):
    """The batch's matrices and the right-hand sides of all of them in one allocation, each at a 256-byte boundary."""
    specs = _batch(case)
    crs = [_crs(dict(family="banded", n=n, width=w, lo=10, hi=60), seed * 131 + i, torch.float32)
           for i, (n, w, _) in enumerate(specs)]
    room = sum((n * k + 63) // 64 * 64 for n, _, k in specs)
    flat = torch.randn(room, generator=_gen(seed + 5), device=CARD)
    return specs, crs, flat


def _views(flat, specs):
    out, at = [], 0
    for n, _, k in specs:
        out.append(flat[at:at + n * k].view(n, k))
        at += (n * k + 63) // 64 * 64
    return out


# ------------------------------------------------------------------ the network
def _training(case, seed):
    """Inputs, targets and the optimiser's state some way into a training."""
    B, nh, g = case["batch"], case["nh"], _gen(seed)
    nin, nout = b.NFEAT, b.SEL_CHOICES

    def normal(*shape, scale=1.0):
        return torch.randn(*shape, generator=g, device=CARD) * scale

    parts = [normal(nh, nin, scale=math.sqrt(2 / nin)), normal(nh, scale=0.1),
             normal(nh, nh, scale=math.sqrt(2 / nh)), normal(nh, scale=0.1),
             normal(nout, nh, scale=math.sqrt(1 / nh)), normal(nout, scale=0.1)]
    P = torch.cat([p.reshape(-1) for p in parts])
    return dict(X=normal(B, nin), T=torch.rand(B, nout, generator=g, device=CARD), P=P, m=normal(P.numel(), scale=1e-3),
                v=torch.rand(P.numel(), generator=g, device=CARD) * 1e-5 + 1e-6)


# ------------------------------------------------------------------ the passes
def prepare(case, seed):
    kind = case["kind"]
    if kind == "train":
        s = _training(case, seed)
        B, nh, nout, P = case["batch"], case["nh"], b.SEL_CHOICES, s["P"]
        return dict(case=case, **s, acts=torch.empty(B * (4 * nh + nout), device=CARD), grads=torch.empty_like(P),
                    scratch=torch.empty(B * (nout + 2 * nh), device=CARD), loss=torch.empty(1, device=CARD))
    if kind == "spmm":
        specs, crs, flat = _batch_data(case, seed)
        mats = [b.cmrs_from_csr(rp, ci, va, n, case["height"], dtype=b.CMRS_F32) for n, rp, ci, va in crs]
        Y = torch.zeros_like(flat)
        plan = b.SpmmPlan(mats, _views(flat, specs), _views(Y, specs))
        return dict(case=case, plan=plan, Y=Y)
    n, rp, ci, va = _crs(case, seed, _input_type(case))
    if kind in ("pad", "sort"):
        return dict(case=case, rp=rp, ci=ci, va=va, n=n)
    x = _vector(n, seed, _input_type(case))
    if kind == "setup":
        path = os.path.join(os.path.dirname(os.path.abspath(b.__file__)), "data", "selector_model.npz")
        return dict(case=case, rp=rp, ci=ci, va=va, n=n, x=x, model=selector.load_model(path))
    flags = b.CMRS_SORTED if case["form"] == "sorted" else 0
    A = b.cmrs_from_csr(rp, ci, va, n, case["height"], flags=flags, dtype=b.DTYPES[case["dtype"]])
    if case["form"] == "padded":
        A = b.cmrs_pad(A, case["slots"])
    return dict(case=case, A=A, x=x, y=torch.empty_like(x))


def run(s):
    case = s["case"]
    kind = case["kind"]
    if kind == "spmv":
        return b.cmrs_spmv(s["A"], s["x"], s["y"])
    if kind == "spmm":
        b.cmrs_spmm_batched(s["plan"])
        return s["Y"]
    if kind == "pad":
        A = b.cmrs_from_csr(s["rp"], s["ci"], s["va"], s["n"], case["height"], dtype=b.DTYPES[case["dtype"]])
        A = b.cmrs_pad(A, case["slots"])
        return [A.strip_ptr, A.col_packed, b.stored_values(A)]
    if kind == "sort":
        A = b.cmrs_from_csr(s["rp"], s["ci"], s["va"], s["n"], case["height"], flags=b.CMRS_SORTED,
                            dtype=b.DTYPES[case["dtype"]])
        rp, ci, _ = b.cmrs_to_csr(A)
        return [A.strip_ptr, A.col_packed, b.stored_values(A), rp, ci]
    if kind == "setup":
        h, variant, slots = b.cmrs_select_strip(s["rp"], s["ci"], s["n"], s["model"])
        A = b.cmrs_from_csr(s["rp"], s["ci"], s["va"], s["n"], h, dtype=b.DTYPES[case["dtype"]])
        if slots:
            A = b.cmrs_pad(A, slots)
        return [h, variant, slots, b.cmrs_spmv(A, s["x"], variant=variant)]
    nh, nout, B = case["nh"], b.SEL_CHOICES, case["batch"]
    b.cmrs_mlp_forward(s["X"], s["P"], nh, nout, s["acts"])
    b.cmrs_mlp_backward(s["X"], s["T"], s["P"], s["acts"], nh, nout, s["grads"], s["scratch"], s["loss"])
    b.cmrs_mlp_adam(s["P"], s["grads"], s["m"], s["v"], 500, 2e-3)
    return dict(out=b.mlp_output(s["acts"], B, nh, nout), grads=s["grads"], loss=s["loss"], P=s["P"], m=s["m"],
                v=s["v"])


# ------------------------------------------------------------------ what a pass cannot do without
def work(case):
    kind = case["kind"]
    if kind == "train":
        B, nh, nin, nout = case["batch"], case["nh"], 32, 21
        weights = nh * nin + nh * nh + nout * nh
        params = weights + 2 * nh + nout
        # batch read, outputs and gradients written, parameters and both moments read and written
        return dict(bytes=4 * (B * (nin + 2 * nout) + 7 * params), flops=6 * B * weights - 2 * B * nh * nin + 12 * params)
    if kind == "spmm":
        specs = _batch(case)
        entries = [35 * n for n, _, _ in specs]
        return dict(bytes=sum(8 * e + 4 * n + 8 * n * k for e, (n, _, k) in zip(entries, specs)),
                    flops=sum(2 * e * k for e, (_, _, k) in zip(entries, specs)))
    rows, nnz = _rows(case), _nnz(case)
    sv, sx = VALUE_BYTES[case["dtype"]], 8 if case["dtype"] == "f64" else 4
    crs = nnz * (4 + sx) + 4 * (rows + 1)
    if kind == "setup":
        return dict(bytes=crs + nnz * (4 + sv) + 2 * sx * rows, flops=2 * nnz)
    cmrs = nnz * (4 + sv) + 4 * (-(-rows // case["height"]) + 1)
    if kind == "pad":
        return dict(bytes=crs + cmrs, flops=0)
    if kind == "sort":
        return dict(bytes=crs + 2 * cmrs + nnz * (4 + sv) + 4 * (rows + 1), flops=0)
    return dict(bytes=cmrs + 2 * sx * rows, flops=2 * nnz)


# ------------------------------------------------------------------ the same in 64 bits
def _product(n, rp, ci, va, x):
    A = torch.sparse_csr_tensor(rp.to(torch.int64), ci.to(torch.int64), va.double(), size=(n, x.shape[0]))
    return A @ x.double()


def _packed(n, rp, ci, height):
    """Strip pointer, strip of each entry and packed words of the CRS matrix."""
    bits = max(4, (height - 1).bit_length())
    strips = -(-n // height)
    sp = rp[torch.arange(strips + 1, device=CARD).mul(height).clamp(max=n)]
    row = torch.repeat_interleave(torch.arange(n, device=CARD), (rp[1:] - rp[:-1]).to(torch.int64))
    word = (ci.to(torch.int64) << bits) | (row % height)
    return sp, row // height, torch.where(word >= 2**31, word - 2**32, word).to(torch.int32)


def exact(case, seed):
    kind = case["kind"]
    if kind == "train":
        s = {k: t.double() for k, t in _training(case, seed).items()}
        B, nh, nin, nout = case["batch"], case["nh"], b.NFEAT, b.SEL_CHOICES
        W1, b1, W2, b2, W3, b3 = torch.split(s["P"], [nh * nin, nh, nh * nh, nh, nout * nh, nout])
        W1, W2, W3 = W1.view(nh, nin), W2.view(nh, nh), W3.view(nout, nh)
        Z1 = s["X"] @ W1.t() + b1
        Z2 = Z1.relu() @ W2.t() + b2
        out = Z2.relu() @ W3.t() + b3
        gO = (out - s["T"]) / (B * nout)
        g2 = (gO @ W3) * (Z2 > 0)
        g1 = (g2 @ W2) * (Z1 > 0)
        grads = torch.cat([t.reshape(-1) for t in (g1.t() @ s["X"], g1.sum(0), g2.t() @ Z1.relu(), g2.sum(0),
                                                   gO.t() @ Z2.relu(), gO.sum(0))])
        m = 0.9 * s["m"] + 0.1 * grads
        v = 0.999 * s["v"] + 0.001 * grads * grads
        P = s["P"] - 2e-3 * (m / (1 - 0.9**500)) / ((v / (1 - 0.999**500)).sqrt() + 1e-8)
        return dict(out=out, grads=grads, loss=((out - s["T"]) ** 2).sum().reshape(1) / (2 * B * nout), P=P, m=m, v=v)
    if kind == "spmm":
        specs, crs, flat = _batch_data(case, seed)
        Y = torch.zeros_like(flat, dtype=torch.float64)
        for (n, rp, ci, va), X, y in zip(crs, _views(flat, specs), _views(Y, specs)):
            y.copy_(_product(n, rp, ci, va, X))
        return Y
    n, rp, ci, va = _crs(case, seed, _input_type(case))
    if kind == "spmv":
        return _product(n, rp, ci, va, _vector(n, seed, _input_type(case)).view(-1, 1)).view(-1)
    if kind == "setup":
        return [None, None, None, _product(n, rp, ci, va, _vector(n, seed, va.dtype).view(-1, 1)).view(-1)]
    if kind == "sort" and case["dtype"] in ("f64", "f32"):
        sp, strip, word = _packed(n, rp, ci, case["height"])
        order = torch.sort(strip * n + ci.to(torch.int64), stable=True)[1]
        return [sp, word[order], va[order].double(), rp, ci]
    return None
