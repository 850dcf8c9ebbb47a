"""The calls whose time counts: RU-QLP decompositions and the steps a program
calls by themselves (products with A, orthonormalisation), over the sizes of
the paper's workloads.  Every pass goes through ``ruqlp.Handle``.  The
large BF16 decomposition is listed by the two steps it repeats (a pass over A
and the orthonormalisation of its result)."""
from __future__ import annotations

import math

import torch

from paper_2209_12464_gb300 import ruqlp

DTYPES = {"f64": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16}
_handle = None


def _h():
    """The process's handle, as a program keeps one: its workspace and plans
    serve every call."""
    global _handle
    if _handle is None:
        _handle = ruqlp.Handle(0, torch.cuda.current_stream().cuda_stream)
    return _handle


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------
def listed():
    return [
        # the plain form, everything in FP64: one small dense matrix (latency,
        # FP64 arithmetic)
        dict(name="plain_f64", kind="decompose", dtype="f64", m=1000, n=800, k=20, p=10, q=1,
             finish=0),
        # the largest matrix of the batched mix, alone, in FP32, with the
        # paper's last step (the QR of L, whose diagonal are the L-values)
        dict(name="dense_f32", kind="decompose", dtype="f32", m=4096, n=2048, k=64, p=8, q=1,
             finish=1),
        # the batched workload: 512 matrices of uneven shapes, BF16 through
        # the tensor cores
        dict(name="batch_bf16", kind="batch", dtype="bf16", count=512, p=8, q=1, shapes=4),
        # a batch as the request loop forms them (at most 64 matrices), FP32
        dict(name="batch_f32", kind="batch", dtype="f32", count=64, p=8, q=1, shapes=9),
        # the sparse workload: 0.1 % density with a planted rank-100 term
        dict(name="csr_bf16", kind="csr", dtype="bf16", m=200000, n=100000, per_row=100, k=100,
             p=10, q=1),
        # one pass over the large dense matrix, the step a decomposition
        # repeats 2 q + 2 times: BF16 sketch, A times a Gaussian matrix
        dict(name="sketch_bf16", kind="sketch", dtype="bf16", m=20000, n=20000, d=220, trans=0),
        # the transposed pass of the large served matrices (wider than one
        # tensor-core tile: two column chunks)
        dict(name="sketch_bf16_t", kind="sketch", dtype="bf16", m=16384, n=8192, d=272, trans=1),
        # the same large matrix kept in FP32: the transposed pass
        dict(name="sketch_f32_t", kind="sketch", dtype="f32", m=20000, n=20000, d=220, trans=1),
        # a small FP32 sketch of ragged sizes (rows not on 16-byte boundaries)
        dict(name="sketch_f32_small", kind="sketch", dtype="f32", m=1001, n=777, d=37, trans=0),
        # an FP64 pass at a width that is no multiple of a tile
        dict(name="sketch_f64", kind="sketch", dtype="f64", m=8192, n=4096, d=72, trans=0),
        # orthonormalising the large matrix's sketch, done after every pass
        dict(name="orth_f32", kind="orth", dtype="f32", m=20000, d=220),
        # the smallest call: an orthonormal basis of a small sketch (latency)
        dict(name="orth_f32_small", kind="orth", dtype="f32", m=1000, d=30),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the ranges above: dense matrices from the batched mix's
    smallest to 20000 x 20000, sketches of 16 to 272 columns."""
    kind = rng.choice(("decompose", "decompose", "batch", "csr", "sketch", "sketch", "sketch",
                       "sketch", "orth", "orth"))
    if kind == "decompose":
        m, n = _log(rng, 256, 4096), _log(rng, 128, 2048)
        return dict(kind=kind, dtype=rng.choice(("f64", "f32")), m=m, n=n, k=rng.randint(8, 64),
                    p=rng.choice((8, 10, 16)), q=rng.choice((0, 1, 1, 2)),
                    finish=rng.choice((0, 0, 1)))
    if kind == "batch":
        return dict(kind=kind, dtype=rng.choice(("bf16", "f32")), count=_log(rng, 4, 256), p=8,
                    q=rng.choice((0, 1, 1, 2)), shapes=rng.randint(10, 1 << 20))
    if kind == "csr":
        m = _log(rng, 20000, 200000)
        return dict(kind=kind, dtype=rng.choice(("bf16", "f32")), m=m, n=m // rng.choice((1, 2, 3)),
                    per_row=rng.randint(40, 100), k=rng.randint(16, 100), p=rng.choice((8, 10)),
                    q=rng.choice((0, 1)))
    if kind == "sketch":
        dtype, trans = rng.choice(("bf16", "bf16", "f32", "f32", "f64")), rng.randint(0, 1)
        hi = 8192 if dtype == "f64" else 20000
        d = _log(rng, 16, 128 if dtype == "f64" else 272)
        m, n = _log(rng, 300, hi), _log(rng, 300, hi)
        if dtype == "f64":
            n = min(n, 8192 * 4096 * 72 // (m * d))
        if dtype == "bf16" and rng.random() < 0.75:
            n = n // 8 * 8  # mostly rows that start on 16 bytes
        return dict(kind=kind, dtype=dtype, m=m, n=max(n, 300), d=d, trans=trans)
    dtype = rng.choice(("f32", "f32", "f64"))
    d = _log(rng, 16, 128 if dtype == "f64" else 272)
    return dict(kind=kind, dtype=dtype, m=_log(rng, 2 * d, 20000 if dtype == "f64" else 100000),
                d=d)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------
def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed))
    return g


def _orthonormal(g, rows, r):
    """rows x r with orthonormal columns (Haar: the QR of a Gaussian matrix by
    its Cholesky factor), FP32."""
    X = torch.randn(rows, r, generator=g, device="cuda", dtype=torch.float64 if rows * r < 1 << 21
                    else torch.float32)
    for _ in range(2):
        C = torch.linalg.cholesky(X.T.double() @ X.double() if rows * r < 1 << 21
                                  else (X.T @ X).double())
        X = torch.linalg.solve_triangular(C.to(X.dtype), X.T, upper=False).T
    return X.float()


def _spectrum(r, k):
    """1 (k times), then 1/2, 1/3, ...: the slow decay of the paper's
    experiments (Section V-B)."""
    i = torch.arange(r, device="cuda", dtype=torch.float32)
    return torch.where(i < k, torch.ones_like(i), 1.0 / (i - k + 2).clamp(min=1))


def _dense(g, m, n, k, dtype):
    """m x n with that spectrum (its first terms) and a little noise; rows on
    16-byte boundaries where n allows."""
    r = min(m, n, 2 * k + 32)
    U, V = _orthonormal(g, m, r), _orthonormal(g, n, r)
    A = (U * _spectrum(r, k)) @ V.T
    if m * n <= 1 << 28:
        A += 1e-6 * torch.randn(m, n, generator=g, device="cuda")
    return A.to(dtype)


def _shapes(case):
    """The batched mix: m and n log-uniform over [256, 4096] and [128, 2048],
    k uniform over [8, 64]; every size odd or even as it comes."""
    import numpy as np
    rng, out = np.random.default_rng(case["shapes"]), []
    for _ in range(case["count"]):
        m = int(round(math.exp(rng.uniform(math.log(256), math.log(4096)))))
        n = int(round(math.exp(rng.uniform(math.log(128), math.log(2048)))))
        k = int(rng.integers(8, 65))
        out.append((m, n, min(k, n - case["p"] - 1, m - case["p"])))
    return out


def _padded(n, dtype):
    per = 16 // torch.empty((), dtype=dtype).element_size()
    return (n + per - 1) // per * per


def _batch_inputs(case, seed):
    g, dt, p = _gen(seed), DTYPES[case["dtype"]], case["p"]
    As, oms = [], []
    # A_i = U_i S V_i^T with near-orthonormal Gaussian U_i, V_i
    for m, n, k in _shapes(case):
        r = min(m, n, 2 * k + 16)
        U = torch.randn(m, r, generator=g, device="cuda") / math.sqrt(m)
        V = torch.randn(n, r, generator=g, device="cuda") / math.sqrt(n)
        buf = torch.zeros(m, _padded(n, dt), dtype=dt, device="cuda")
        buf[:, :n] = (U * _spectrum(r, k)) @ V.T
        As.append(buf[:, :n])
        oms.append(torch.randn(n, k + p, generator=g, device="cuda", dtype=torch.float64))
    return As, oms


def _csr_inputs(case, seed):
    """Uniform pattern (per_row nonzeros a row on average), values N(0,1) plus
    a planted rank-100 term of scale 10."""
    g, m, n = _gen(seed), case["m"], case["n"]
    nnz, rank = m * case["per_row"], 100
    key = torch.unique(torch.randint(0, m * n, (nnz,), generator=g, device="cuda"))
    rows, cols = key // n, key % n
    rowptr = torch.zeros(m + 1, dtype=torch.int64, device="cuda")
    rowptr[1:] = torch.cumsum(torch.bincount(rows, minlength=m), 0)
    vals = torch.randn(key.numel(), generator=g, device="cuda")
    X = torch.randn(m, rank, generator=g, device="cuda")
    Y = torch.randn(n, rank, generator=g, device="cuda")
    for a in range(0, key.numel(), 1 << 21):
        s = slice(a, a + (1 << 21))
        vals[s] += 10 / math.sqrt(rank) * (X[rows[s]] * Y[cols[s]]).sum(1)
    om = torch.randn(n, case["k"] + case["p"], generator=g, device="cuda", dtype=torch.float64)
    return rowptr.int(), cols.int(), vals.to(DTYPES[case["dtype"]]), om


def _sketch_inputs(case, seed):
    g, dt, d = _gen(seed), DTYPES[case["dtype"]], case["d"]
    m, n = case["m"], case["n"]
    wt = torch.float64 if case["dtype"] == "f64" else torch.float32
    A = _dense(g, m, n, max(1, int(d * 0.9)), dt)
    if case["trans"]:  # A^T Q with an orthonormal basis Q
        X = torch.randn(m, d, generator=g, device="cuda", dtype=wt) / math.sqrt(m)
    else:              # A Omega
        X = torch.randn(n, d, generator=g, device="cuda", dtype=wt)
    return A, X


def _orth_input(case, seed):
    """A sketch Y = A Omega of a matrix with the slow-decay spectrum."""
    g, M, d = _gen(seed), case["m"], case["d"]
    r = min(M, 2 * d)
    Y = (_orthonormal(g, M, r) * _spectrum(r, max(1, int(d * 0.9)))) @ torch.randn(
        r, d, generator=g, device="cuda")
    return Y.to(DTYPES[case["dtype"]])


def _decompose_inputs(case, seed):
    g = _gen(seed)
    A = _dense(g, case["m"], case["n"], case["k"], DTYPES[case["dtype"]])
    om = torch.randn(case["n"], case["k"] + case["p"], generator=g, device="cuda",
                     dtype=torch.float64)
    return A, om


def prepare(case, seed):
    kind, h = case["kind"], _h()
    if kind == "batch":
        As, oms = _batch_inputs(case, seed)
        shapes, p = _shapes(case), case["p"]
        # the outputs packed one after another, as a program that copies them
        # on in one piece keeps them
        size = [(m * (k + p), (k + p) ** 2, n * (k + p)) for m, n, k in shapes]
        step = [[(x + 3) // 4 * 4 for x in s] for s in size]
        packs = [torch.zeros(sum(s[j] for s in step), device="cuda") for j in range(3)]
        outs, at = [], [0, 0, 0]
        for (m, n, k), s, t in zip(shapes, size, step):
            dims = ((m, k + p), (k + p, k + p), (n, k + p))
            outs.append(tuple(packs[j][at[j]:at[j] + s[j]].view(dims[j]) for j in range(3)))
            at = [a + x for a, x in zip(at, t)]
        b = h.prepare_batch(As, oms, [k for _, _, k in shapes], p, case["q"], outs=outs)
        return dict(case=case, batch=b, packs=packs)
    make = {"decompose": _decompose_inputs, "csr": _csr_inputs, "sketch": _sketch_inputs,
            "orth": lambda c, s: (_orth_input(c, s),)}[kind]
    return dict(case=case, args=make(case, seed))


def run(state):
    c, h = state["case"], _h()
    if c["kind"] == "decompose":
        A, om = state["args"]
        return h.decompose(A, om, c["k"], c["p"], c["q"], finish_paper=c["finish"])
    if c["kind"] == "batch":
        flags = state["batch"].run()
        return dict(zip("QLP", state["packs"]), flags=torch.tensor(flags))
    if c["kind"] == "csr":
        rowptr, cols, vals, om = state["args"]
        return h.decompose_csr(rowptr, cols, vals, (c["m"], c["n"]), om, c["k"], c["p"], c["q"])
    if c["kind"] == "sketch":
        return h.sketch(*state["args"], trans=bool(c["trans"]))
    return h.orth(*state["args"])


# ---------------------------------------------------------------------------
# work and exact results
# ---------------------------------------------------------------------------
def work(case):
    es = {"f64": 8, "f32": 4, "bf16": 2}[case["dtype"]]
    ws = 8 if case["dtype"] == "f64" else 4

    def qlp(m, n, nnz, abytes, d, q):
        out = ws * (m * d + d * d + n * d)
        # 2 q + 2 passes over A; per pass a Gram and a triangular solve
        return abytes + 8 * n * d + out, (2 * q + 2) * 2 * nnz * d + (q + 1) * (m + n) * 2 * d * d

    if case["kind"] == "sketch":
        m, n, d = case["m"], case["n"], case["d"]
        return {"bytes": m * n * es + (m + n) * d * ws, "flops": 2 * m * n * d}
    if case["kind"] == "orth":
        return {"bytes": 2 * case["m"] * case["d"] * ws, "flops": 2 * case["m"] * case["d"] ** 2}
    if case["kind"] == "batch":
        w = [qlp(m, n, m * n, m * n * es, k + case["p"], case["q"]) for m, n, k in _shapes(case)]
        return {"bytes": sum(x for x, _ in w), "flops": sum(x for _, x in w)}
    m, n, d = case["m"], case["n"], case["k"] + case["p"]
    if case["kind"] == "csr":
        nnz = m * case["per_row"]
        b, f = qlp(m, n, nnz, nnz * (es + 4) + 4 * (m + 1), d, case["q"])
    else:
        b, f = qlp(m, n, m * n, m * n * es, d, case["q"])
    return {"bytes": b, "flops": f}


def _qr(Y):
    """Thin QR with a non-negative diagonal of R."""
    Q, R = torch.linalg.qr(Y)
    s = torch.where(torch.diagonal(R) < 0, -1.0, 1.0).to(Y.dtype)
    return Q * s, R * s[:, None]


def _qlp(mul, tmul, om, q, finish):
    """Algorithm 1 + 2 in FP64: A ~= Q L P^T."""
    Q = _qr(mul(om))[0]
    for _ in range(q):
        Q = _qr(mul(_qr(tmul(Q))[0]))[0]
    P, R = _qr(tmul(Q))
    L = R.T
    if finish:
        Pt, L = _qr(L)
        Q = Q @ Pt
    return Q, L, P


def exact(case, seed):
    if case["kind"] == "sketch":
        A, X = _sketch_inputs(case, seed)
        if case["dtype"] == "bf16":  # the entry point takes X in BF16
            X = X.bfloat16()
        A, X = A.double(), X.double()
        return (A.T if case["trans"] else A) @ X
    if case["kind"] == "orth":
        return _qr(_orth_input(case, seed).double())[0]
    if case["kind"] == "decompose":
        A, om = _decompose_inputs(case, seed)
        A = A.double()
        Q, L, P = _qlp(lambda x: A @ x, lambda y: A.T @ y, om, case["q"], case["finish"])
        return Q, L, P, None
    if case["kind"] == "csr":
        rowptr, cols, vals, om = _csr_inputs(case, seed)
        m, n = case["m"], case["n"]
        rows = torch.repeat_interleave(torch.arange(m, device="cuda"), rowptr.diff().long())
        A = torch.sparse_csr_tensor(rowptr, cols, vals.double(), size=(m, n))
        order = torch.argsort(cols.long() * m + rows)
        colptr = torch.zeros(n + 1, dtype=torch.int32, device="cuda")
        colptr[1:] = torch.cumsum(torch.bincount(cols.long(), minlength=n), 0)
        At = torch.sparse_csr_tensor(colptr, rows[order].int(), vals[order].double(), size=(n, m))
        Q, L, P = _qlp(lambda x: A @ x, lambda y: At @ y, om, case["q"], 0)
        return Q, L, P, None
    # batches: FP32 in full; BF16 the middle factors alone (the BF16 operands
    # of the passes turn the bases by more than any later rounding)
    As, oms = _batch_inputs(case, seed)
    packs = ([], [], [])
    for A, om in zip(As, oms):
        A = A.double()
        if case["dtype"] == "bf16":
            om = om.bfloat16().double()
        for out, x in zip(packs, _qlp(lambda x: A @ x, lambda y: A.T @ y, om, case["q"], 0)):
            out.append(torch.nn.functional.pad(x.reshape(-1), (0, -x.numel() % 4)))
    Q, L, P = (torch.cat(x) for x in packs)
    if case["dtype"] == "bf16":
        Q = P = None
    return dict(Q=Q, L=L, P=P, flags=None)
