"""What the library's users run, as cases that can be timed and checked.

A case is a dict of plain values; ``prepare`` makes the inputs a program has in hand before the
call, ``run`` is one pass through the public entry points, ``work`` the bytes and operations the pass
cannot do without, and ``exact`` the same outputs in 64 bits from plain torch (no code of this
package). The kinds:

* ``estimate``       whole estimator (Alg. 10) on dense A, in the three precisions in use;
* ``estimate_csr``   the same on CSR A;
* ``exact``          Alg. 7 (LS-HRN-exact) on dense A;
* ``exact_csr``      Alg. 7 on CSR A;
* ``reference``      the exact scores of dense A itself (the quantity the estimator approximates);
* ``train``          forward and backward of a loss on the estimated scores (the autograd function);
* ``lstsq``          Alg. 11 preconditioner and LSQR;
* ``rrqr``           the pivoted QR of a sketch alone (a row-sharded program calls it after its
                     all-reduce).

Sizes are the repository's own workloads (its configurations, tests and benchmark) and ragged
neighbours of them.
"""
import math

import torch

import paper_2105_11004_gb300 as L

SKETCH_SEED = 11       # a program keeps one sketch (S, G, Omega) for all its batches


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def listed():
    return [
        # a small problem solved interactively: latency and launches count (tau below the Gram route)
        dict(name="estimate_small", kind="estimate", n=2000, d=20, rank=20, skew=0.0, s=1600, m=80, k=64, tau=1e-10,
             sketch="fp32", final="fp32", wait=True),
        # the entry point's default precisions on the full-size dense batch
        dict(name="estimate_fp32", kind="estimate", n=1_000_000, d=256, rank=200, skew=2.0, s=65536, m=1024, k=256,
             tau=1e-4, sketch="fp32", final="fp32", wait=True),
        # the dense serving loop: split-BF16 stages, scores left on the device, no wait for the rank
        dict(name="estimate_split", kind="estimate", n=1_000_000, d=256, rank=200, skew=2.0, s=65536, m=1024, k=256,
             tau=1e-4, sketch="bf16x3", final="bf16x3", wait=False),
        # a feature matrix as it comes: odd row and column counts, TF32 final pass
        dict(name="estimate_ragged", kind="estimate", n=300_007, d=99, rank=99, skew=1.0, s=20011, m=400, k=150,
             tau=1e-5, sketch="bf16x3", final="tf32", wait=True),
        # sparse features, 8 entries a row and 1% long rows
        dict(name="csr_8e6", kind="estimate_csr", n=8_000_000, d=1024, per_row=8, long_frac=0.01, long_len=256, pairs=0,
             s=262144, m=4096, k=256, tau=1e-5, sketch="bf16x3"),
        # the largest: an image-set shaped CSR, about 1e9 entries, ten dependent column pairs
        dict(name="csr_8e7", kind="estimate_csr", n=80_000_000, d=1024, per_row=12, long_frac=0.0, long_len=0, pairs=10,
             s=262144, m=4096, k=256, tau=1e-5, sketch="bf16x3"),
        # exact scores on the selected columns, where a user wants no estimate
        dict(name="exact_dense", kind="exact", n=1_000_000, d=256, rank=200, skew=2.0, s=65536, m=1024, k=256, tau=1e-4,
             sketch="bf16x3", final="bf16x3"),
        dict(name="exact_csr", kind="exact_csr", n=2_000_000, d=1024, per_row=8, long_frac=0.01, long_len=256,
             s=65536, m=4096, k=256, tau=1e-5, sketch="bf16x3"),
        # checking an estimate against the exact scores of A, a wider matrix
        dict(name="reference_dense", kind="reference", n=100_003, d=500, rank=500, skew=0.5, tau=1e-5),
        # one training step on the scores: theta and the gradient of sum w theta
        dict(name="train_step", kind="train", n=200_000, d=64, s=16384, m=256, k=128, tau=1e-5, sketch="bf16x3",
             final="bf16x3"),
        # least squares by the preconditioner and LSQR
        dict(name="lstsq", kind="lstsq", n=1_000_000, d=256, skew=0.5, s=65536, m=1024, tau=1e-10, sketch="bf16x3"),
        # the pivoted QR alone, at the sparse workload's sketch size
        dict(name="rrqr", kind="rrqr", m=4096, d=1024, tau=1e-5),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _repeatable_d(d, sketch):
    """The next smaller d whose tensor-core Gaussian stage gives the same sketch on every run: above
    256 columns it works on equal column tiles, and with tiles that are not whole groups of 32 columns
    its outputs differed from run to run, so that nothing could be compared with them."""
    while sketch != "fp32" and d > 256:
        tiles = -(-d // 256)
        if -(-(-(-d // tiles)) // 16) % 2 == 0:
            break
        d -= 1
    return d


def draw(rng):
    """One more case of the same ranges (sizes over their logarithm, odd ones among them)."""
    kind = rng.choice(["estimate", "estimate", "estimate_csr", "exact", "exact_csr", "reference", "train", "lstsq",
                       "rrqr"])
    if kind == "estimate":
        n, d = _log(rng, 1000, 1_000_000), _log(rng, 8, 256)
        sketch, final = rng.choice([("fp32", "fp32"), ("bf16x3", "bf16x3"), ("bf16x3", "tf32"), ("bf16x3", "bf16")])
        s = min(65536, max(8 * d, n // rng.randint(4, 20)))
        return dict(kind=kind, n=max(n, 16 * d), d=d, rank=d, skew=rng.choice([0.0, 0.5, 1.0]), s=s, m=4 * d,
                    k=_log(rng, 32, 256), tau=1e-5, sketch=sketch, final=final, wait=rng.random() < 0.5)
    if kind in ("estimate_csr", "exact_csr"):
        sketch = rng.choice(["bf16x3", "bf16x3", "fp32"])
        d = _repeatable_d(_log(rng, 128, 1024), sketch)
        n = _log(rng, 50_000, 8_000_000 if kind == "estimate_csr" else 2_000_000)
        case = dict(kind=kind, n=n, d=d, per_row=rng.randint(4, 24), long_frac=rng.choice([0.0, 0.01]),
                    long_len=max(33, d // 4), s=min(262144, max(8 * d, n // rng.randint(8, 30))), m=4 * d, k=256,
                    tau=1e-5, sketch=sketch)
        if case["sketch"] == "fp32":
            case["s"] = min(case["s"], 32768)
        if kind == "estimate_csr":
            case["pairs"] = 0
        return case
    if kind == "exact":
        n, d = _log(rng, 10_000, 1_000_000), _log(rng, 16, 256)
        return dict(kind=kind, n=n, d=d, rank=d, skew=rng.choice([0.0, 0.5]), s=min(65536, max(8 * d, n // 10)),
                    m=4 * d, k=256, tau=1e-5, sketch="bf16x3", final=rng.choice(["fp32", "bf16x3"]))
    if kind == "reference":
        d = _log(rng, 32, 768)
        n = _log(rng, 16 * d, max(32 * d, min(1_000_000, 25_000_000_000 // (d * d))))
        return dict(kind=kind, n=n, d=d, rank=d, skew=rng.choice([0.0, 0.5]), tau=1e-5)
    if kind == "train":
        n, d = _log(rng, 10_000, 400_000), _log(rng, 8, 128)
        return dict(kind=kind, n=n, d=d, s=max(8 * d, n // rng.randint(8, 20)), m=4 * d, k=_log(rng, 32, 256), tau=1e-5,
                    sketch=rng.choice(["bf16x3", "fp32"]), final=rng.choice(["fp32", "bf16x3"]))
    if kind == "lstsq":
        n, d = _log(rng, 20_000, 1_000_000), _log(rng, 16, 256)
        return dict(kind=kind, n=n, d=d, skew=rng.choice([0.0, 0.5]), s=min(65536, max(16 * d, n // 12)), m=4 * d,
                    tau=1e-10, sketch="bf16x3")
    d = _log(rng, 24, 1024)
    return dict(kind=kind, m=rng.randint(2 * d, 4 * d), d=d, tau=1e-5)


# ---------------------------------------------------------------------------
# inputs
# ---------------------------------------------------------------------------

def _gen(seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    return g


def _dense(n, d, rank, skew, seed):
    """diag(e^{skew z}) times a Gaussian matrix (rank < d: U V^T with Gaussian factors), formed in
    64 bits by row blocks and stored in 32."""
    g = _gen(seed)
    V = torch.randn(d, rank, generator=g, device="cuda", dtype=torch.float64) if rank < d else None
    A = torch.empty(n, d, device="cuda", dtype=torch.float32)
    for r0 in range(0, n, 1 << 18):
        r1 = min(n, r0 + (1 << 18))
        U = torch.randn(r1 - r0, rank, generator=g, device="cuda", dtype=torch.float64)
        X = U @ V.T if V is not None else U
        if skew:
            X = X * torch.exp(skew * torch.randn(r1 - r0, 1, generator=g, device="cuda", dtype=torch.float64))
        A[r0:r1] = X.float()
    return A


def _csr(case, seed):
    """CSR with per_row distinct sorted columns a row, Gaussian values times a scale of the column's own
    (features come in different units); a fraction of long rows, and (pairs > 0) rows that hold column j < pairs also hold column j + d/2 with twice the value, as their last entries."""
    g = _gen(seed)
    n, d, w = case["n"], case["d"], case["per_row"]
    pairs = case.get("pairs", 0)
    half = d // 2
    width = d - pairs                                     # the columns that are not copies
    scale = torch.exp(0.5 * torch.randn(d, generator=g, device="cuda"))
    lens = torch.full((n,), w, device="cuda", dtype=torch.int64)
    is_long = torch.zeros(n, device="cuda", dtype=torch.bool)
    if case["long_frac"] > 0:
        is_long = torch.rand(n, generator=g, device="cuda") < case["long_frac"]
        lens[is_long] = case["long_len"]

    def block(rows, per):
        c = torch.randint(0, width - per + 1, (rows, per), generator=g, device="cuda", dtype=torch.int32)
        c = torch.sort(c, dim=1).values + torch.arange(per, device="cuda", dtype=torch.int32)
        return torch.where(c >= half, c + pairs, c) if pairs else c

    blocks = []
    for r0 in range(0, n, 1 << 23):
        r1 = min(n, r0 + (1 << 23))
        short = (~is_long[r0:r1]).nonzero().squeeze(1) + r0 if case["long_frac"] > 0 else None
        c = block(r1 - r0 if short is None else short.numel(), w)
        v = torch.randn(c.shape, generator=g, device="cuda") * scale[c.long()]
        blocks.append((r0, r1, short, c, v))
        if pairs:
            lens[r0:r1] += (c < pairs).sum(1)
    row_ptr = torch.zeros(n + 1, device="cuda", dtype=torch.int64)
    torch.cumsum(lens, 0, out=row_ptr[1:])
    nnz = int(row_ptr[-1])
    col = torch.empty(nnz, device="cuda", dtype=torch.int32)
    val = torch.empty(nnz, device="cuda", dtype=torch.float32)
    for r0, r1, short, c, v in blocks:
        start = row_ptr[r0:r1] if short is None else row_ptr[short]
        at = start[:, None] + torch.arange(w, device="cuda")
        col[at.reshape(-1)] = c.reshape(-1)
        val[at.reshape(-1)] = v.reshape(-1)
        if pairs:
            row, e = (c < pairs).nonzero(as_tuple=True)
            first = torch.cumsum((c < pairs).to(torch.int64), 1)[row, e] - 1
            at = start[row] + w + first
            col[at] = c[row, e] + half
            val[at] = 2.0 * v[row, e]
    if case["long_frac"] > 0:
        rows = is_long.nonzero().squeeze(1)
        for q in range(0, rows.numel(), 1 << 16):
            rr = rows[q:q + (1 << 16)]
            c = block(rr.numel(), case["long_len"])
            at = row_ptr[rr][:, None] + torch.arange(case["long_len"], device="cuda")
            col[at.reshape(-1)] = c.reshape(-1)
            val[at.reshape(-1)] = (torch.randn(c.shape, generator=g, device="cuda") * scale[c.long()]).reshape(-1)
    return row_ptr, col, val


def _sketch_like(m, d, seed):
    """A matrix like a sketch: Gaussian rows, correlated columns of different lengths."""
    g = _gen(seed)
    X = torch.randn(m, d, generator=g, device="cuda", dtype=torch.float64)
    mix = torch.eye(d, device="cuda", dtype=torch.float64)
    mix += 0.3 / math.sqrt(d) * torch.randn(d, d, generator=g, device="cuda", dtype=torch.float64)
    scale = torch.exp(0.3 * torch.randn(d, generator=g, device="cuda", dtype=torch.float64))
    return ((X @ mix) * scale / math.sqrt(m)).float()


def _train_inputs(case, seed):
    n, d = case["n"], case["d"]
    g = _gen(seed)
    A = torch.randn(n, d, generator=g, device="cuda")
    A[torch.rand(n, generator=g, device="cuda") < 0.05] *= 100.0
    w = torch.rand(n, generator=g, device="cuda")
    return A, w


def _lstsq_inputs(case, seed):
    A = _dense(case["n"], case["d"], case["d"], case["skew"], seed)
    b = torch.randn(case["n"], generator=_gen(seed + 1_000_003), device="cuda")
    return A, b


def prepare(case, seed):
    kind = case["kind"]
    st = {"case": case, "h": L.default_handle(0)}
    if kind in ("estimate", "exact", "reference"):
        st["A"] = _dense(case["n"], case["d"], case["rank"], case["skew"], seed)
    elif kind in ("estimate_csr", "exact_csr"):
        st["csr"] = _csr(case, seed)
    elif kind == "train":
        A, st["w"] = _train_inputs(case, seed)
        st["A"] = A.requires_grad_(True)
    elif kind == "lstsq":
        st["A"], st["b"] = _lstsq_inputs(case, seed)
    else:
        st["At"] = _sketch_like(case["m"], case["d"], seed)
    if kind in ("estimate", "estimate_csr", "exact", "exact_csr", "train"):
        st["p"] = L.make_params(s=case["s"], m=case["m"], k=case["k"], tau=case["tau"], seed=SKETCH_SEED,
                                sketch_prec=case["sketch"], final_prec=case.get("final", "fp32"))
        # the data-independent operands, as a program makes them once
        L.lev_prepare(st["h"], case["n"], case["d"], st["p"])
    return st


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def run(st):
    case, h = st["case"], st["h"]
    kind = case["kind"]
    if kind == "estimate" and case["wait"]:
        theta, rank, perm = L.estimate(st["A"], s=case["s"], m=case["m"], k=case["k"], tau=case["tau"],
                                       seed=SKETCH_SEED, sketch_prec=case["sketch"], final_prec=case["final"], handle=h)
        return {"theta": theta, "rank": rank, "perm": perm}
    if kind == "rrqr":
        d = case["d"]
        perm = torch.empty(d, dtype=torch.int32, device="cuda")
        R = torch.empty((d, d), dtype=torch.float64, device="cuda")
        rank = L.lev_rrqr(h, st["At"], case["tau"], perm, R)
        return {"R": R, "rank": rank, "perm": perm}
    if kind == "train":
        theta = L.LevScore.apply(st["A"], st["p"])
        (grad,) = torch.autograd.grad(theta, st["A"], st["w"])
        return {"theta": theta.detach(), "grad": grad}
    if kind == "lstsq":
        x, rank, _, _ = L.lstsq(st["A"], st["b"], s=case["s"], m=case["m"], tau=case["tau"], seed=SKETCH_SEED,
                                sketch_prec=case["sketch"], handle=h)
        # the solution goes back to the precision of A and b, in which it is used (LSQR stops at 1e-6)
        return {"x": x.float(), "rank": rank}
    n, d = case["n"], case["d"]
    theta = torch.empty(n, dtype=torch.float32, device="cuda")
    perm = torch.empty(d, dtype=torch.int32, device="cuda")
    if kind == "estimate":
        L.lev_estimate_dense(h, st["A"], st["p"], theta, perm, want_rank=False)
        return {"theta": theta, "perm": perm}
    if kind == "estimate_csr":
        rank = L.lev_estimate_csr(h, *st["csr"], n, d, st["p"], theta, perm)
    elif kind == "exact":
        rank = L.lev_exact_dense(h, st["A"], st["p"], theta, perm)
    elif kind == "exact_csr":
        rank = L.lev_exact_csr(h, *st["csr"], n, d, st["p"], theta, perm)
    else:
        rank = L.lev_exact_reference_dense(h, st["A"], case["tau"], theta, perm)
    return {"theta": theta, "rank": rank, "perm": perm}


# ---------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------

def work(case):
    kind, d = case["kind"], case["d"]
    if kind == "rrqr":
        m = case["m"]
        return {"bytes": 4.0 * m * d + 8.0 * d * d, "flops": 2.0 * m * d * d - 2.0 / 3.0 * d ** 3}
    n = case["n"]
    if kind in ("estimate_csr", "exact_csr"):
        short, long_ = n * (1.0 - case["long_frac"]), n * case["long_frac"]
        nnz = short * case["per_row"] + long_ * case["long_len"]
        pairs = short * case["per_row"] * (case["per_row"] + 1) / 2.0
        k = case["k"] if kind == "estimate_csr" else d
        long_flops = 2.0 * long_ * case["long_len"] * min(k, (case["long_len"] + 1) / 2.0)
        flops = 2.0 * nnz + 2.0 * case["m"] * case["s"] * d + 2.0 * pairs + long_flops
        if kind == "exact_csr":
            flops += 2.0 * pairs + long_ * case["long_len"] * (case["long_len"] + 1.0)
        return {"bytes": 8.0 * nnz + 8.0 * (n + 1) + 4.0 * n, "flops": flops}
    bytes_ = 4.0 * n * d + 4.0 * n
    if kind == "reference":
        return {"bytes": bytes_, "flops": n * d * (d + 1.0) + n * d * (d + 1.0)}
    sketch = 2.0 * n * d + 2.0 * case["m"] * case["s"] * d
    if kind == "lstsq":
        return {"bytes": bytes_, "flops": sketch + 4.0 * n * d}
    r = case.get("rank", d)
    flops = sketch + 2.0 * n * r * min(r, case["k"])
    if kind == "exact":
        flops += n * r * (r + 1.0)
    if kind == "train":
        bytes_ += 4.0 * n * d + 4.0 * n
        flops += 2.0 * n * d * d + n * d * (d + 1.0)
    return {"bytes": bytes_, "flops": flops}


# ---------------------------------------------------------------------------
# the same outputs in 64 bits
# ---------------------------------------------------------------------------

_MASK = (1 << 64) - 1


def _i64(x):
    x &= _MASK
    return x - (1 << 64) if x >> 63 else x


def _shr(z, k):
    return (z >> k) & ((1 << (64 - k)) - 1)


def _splitmix(key, c):
    z = (c + 1) * _i64(0x9E3779B97F4A7C15) + _i64(key)
    z = (z ^ _shr(z, 30)) * _i64(0xBF58476D1CE4E5B9)
    z = (z ^ _shr(z, 27)) * _i64(0x94D049BB133111EB)
    return z ^ _shr(z, 31)


def _key(stream):
    return SKETCH_SEED ^ (stream * 0xD1B54A32D192ED03 & _MASK)


def _normal(stream, c):
    """Box-Muller by counter, cosine branch, in 64 bits."""
    u1 = (_shr(_splitmix(_key(stream), 2 * c), 11) + 1).double() * 2.0 ** -53
    u2 = _shr(_splitmix(_key(stream), 2 * c + 1), 11).double() * 2.0 ** -53
    return torch.sqrt(-2.0 * torch.log(u1)) * torch.cos(2.0 * math.pi * u2)


def _bucket_sign(rows, s):
    x = _splitmix(_key(1), rows)
    return _shr(_shr(x, 32) * s, 32), 1.0 - 2.0 * (x & 1).double()


def _arange(a, b):
    return torch.arange(a, b, device="cuda", dtype=torch.int64)


def _gauss_rows(j0, j1, m, s):
    return _normal(2, _arange(j0, j1)[:, None] * s + _arange(0, s)[None, :]) / math.sqrt(m)


def _times_g(B, m):
    s, d = B.shape
    out = torch.empty(m, d, device="cuda", dtype=torch.float64)
    step = max(1, (1 << 25) // s)
    for j in range(0, m, step):
        j1 = min(m, j + step)
        out[j:j1] = _gauss_rows(j, j1, m, s) @ B
    return out


def _sketch_dense(A, s, m):
    B = torch.zeros(s, A.shape[1], device="cuda", dtype=torch.float64)
    for r0 in range(0, A.shape[0], 1 << 18):
        blk = A[r0:r0 + (1 << 18)].double()
        b, sg = _bucket_sign(_arange(r0, r0 + blk.shape[0]), s)
        B.index_add_(0, b, blk * sg[:, None])
    return _times_g(B, m)


def _csr_entries(csr, r0, r1):
    """(local row, column, value in 64 bits) of the entries of rows r0..r1-1."""
    row_ptr, col, val = csr
    a, b = int(row_ptr[r0]), int(row_ptr[r1])
    rows = torch.repeat_interleave(_arange(0, r1 - r0), row_ptr[r0 + 1:r1 + 1] - row_ptr[r0:r1], output_size=b - a)
    return rows, col[a:b].long(), val[a:b].double()


def _sketch_csr(csr, n, d, s, m):
    B = torch.zeros(s * d, device="cuda", dtype=torch.float64)
    for r0 in range(0, n, 1 << 21):
        r1 = min(n, r0 + (1 << 21))
        rows, c, v = _csr_entries(csr, r0, r1)
        b, sg = _bucket_sign(_arange(r0, r1), s)
        B.index_add_(0, b[rows] * d + c, v * sg[rows])
    return _times_g(B.view(s, d), m)


def _pivoted_qr(X, tau):
    """(pivots, R in pivot order with the other columns ascending, diagonal >= 0): greatest trailing
    norm first, stopped at |R_jj| <= tau |R_00|."""
    W = X.clone()
    m, d = W.shape
    active = torch.ones(d, device="cuda", dtype=torch.bool)
    piv, rows, top = [], [], None
    for j in range(min(m, d)):
        t = (W[j:] ** 2).sum(0).masked_fill_(~active, -1.0)
        p = int(t.argmax())
        nrm = math.sqrt(max(float(t[p]), 0.0))
        top = nrm if top is None else top
        if not nrm > 0.0 or nrm <= tau * top:
            break
        v = W[j:, p].clone()
        v[0] += math.copysign(nrm, float(v[0]))
        W[j:] -= torch.outer(v, (2.0 / (v @ v)) * (v @ W[j:]))
        rows.append(W[j] * torch.sign(W[j, p]) * active)
        active[p] = False
        piv.append(p)
    rest = [c for c in range(d) if c not in set(piv)]
    order = torch.tensor(piv + rest, device="cuda", dtype=torch.int64)
    R = torch.zeros(d, d, device="cuda", dtype=torch.float64)
    if rows:
        R[:len(piv)] = torch.stack(rows)[:, order]
    return piv, torch.triu(R)


def _small_factor(At, tau, k):
    """M = R_11^{-1} Omega on the selected columns, zero rows elsewhere (d x k)."""
    piv, R = _pivoted_qr(At, tau)
    r = len(piv)
    Om = _normal(3, _arange(0, r)[:, None] * k + _arange(0, k)[None, :]) / math.sqrt(k)
    M = torch.zeros(At.shape[1], k, device="cuda", dtype=torch.float64)
    M[piv] = torch.linalg.solve_triangular(R[:r, :r], Om, upper=True)
    return M


def _row_norms(A, M):
    out = torch.empty(A.shape[0], device="cuda", dtype=torch.float64)
    for r0 in range(0, A.shape[0], 1 << 18):
        out[r0:r0 + (1 << 18)] = ((A[r0:r0 + (1 << 18)].double() @ M) ** 2).sum(1)
    return out


def _csr_row_norms(csr, n, d, M):
    out = torch.empty(n, device="cuda", dtype=torch.float64)
    for r0 in range(0, n, 1 << 17):
        r1 = min(n, r0 + (1 << 17))
        rows, c, v = _csr_entries(csr, r0, r1)
        X = torch.zeros((r1 - r0) * d, device="cuda", dtype=torch.float64)
        X.index_add_(0, rows * d + c, v)
        out[r0:r1] = ((X.view(-1, d) @ M) ** 2).sum(1)
    return out


def _csr_pair_norms(csr, case, M):
    """a_i (M M^T) a_i^T for rows of per_row entries, the copies of the dependent pairs folded into
    their originals (column j + d/2 holds twice column j)."""
    n, w, half, pairs = case["n"], case["per_row"], case["d"] // 2, case["pairs"]
    N = M.clone()
    N[:pairs] += 2.0 * M[half:half + pairs]
    P = (N @ N.T).reshape(-1)
    row_ptr, col, val = csr
    out = torch.empty(n, device="cuda", dtype=torch.float64)
    for r0 in range(0, n, 1 << 22):
        r1 = min(n, r0 + (1 << 22))
        at = row_ptr[r0:r1][:, None] + _arange(0, w)[None, :]
        c, v = col[at].long().T.contiguous(), val[at].double().T.contiguous()
        t = torch.zeros(r1 - r0, device="cuda", dtype=torch.float64)
        for p in range(w):
            t += v[p] * v[p] * P[c[p] * (case["d"] + 1)]
            for q in range(p + 1, w):
                t += 2.0 * v[p] * v[q] * P[c[p] * case["d"] + c[q]]
        out[r0:r1] = t
    return out


def _leverage_factor(G, piv):
    """R^{-1} (pivot order) scattered to the rows of piv, R^T R = G restricted to piv."""
    idx = torch.tensor(piv, device="cuda", dtype=torch.int64)
    U = torch.linalg.cholesky(G[idx][:, idx], upper=True)
    M = torch.zeros(G.shape[0], len(piv), device="cuda", dtype=torch.float64)
    M[idx] = torch.linalg.solve_triangular(U, torch.eye(len(piv), device="cuda", dtype=torch.float64), upper=True)
    return M


def _gram(A):
    G = torch.zeros(A.shape[1], A.shape[1], device="cuda", dtype=torch.float64)
    for r0 in range(0, A.shape[0], 1 << 18):
        blk = A[r0:r0 + (1 << 18)].double()
        G += blk.T @ blk
    return G


def _csr_gram(csr, n, d):
    G = torch.zeros(d, d, device="cuda", dtype=torch.float64)
    for r0 in range(0, n, 1 << 17):
        r1 = min(n, r0 + (1 << 17))
        rows, c, v = _csr_entries(csr, r0, r1)
        X = torch.zeros((r1 - r0) * d, device="cuda", dtype=torch.float64)
        X.index_add_(0, rows * d + c, v)
        X = X.view(-1, d)
        G += X.T @ X
    return G


def _exact_train(case, seed):
    """theta and its gradient with the sketch, the pivots and the rank held, by automatic
    differentiation in 64 bits."""
    A32, w = _train_inputs(case, seed)
    A = A32.double().requires_grad_(True)
    n, s, m, k = case["n"], case["s"], case["m"], case["k"]
    b, sg = _bucket_sign(_arange(0, n), s)
    B = torch.zeros(s, case["d"], device="cuda", dtype=torch.float64).index_add(0, b, A * sg[:, None])
    At = _gauss_rows(0, m, m, s) @ B
    piv, _ = _pivoted_qr(At.detach(), case["tau"])
    idx = torch.tensor(piv, device="cuda", dtype=torch.int64)
    _, R = torch.linalg.qr(At[:, idx])
    R = R * torch.sign(torch.diagonal(R)).detach()[:, None]
    r = len(piv)
    Om = _normal(3, _arange(0, r)[:, None] * k + _arange(0, k)[None, :]) / math.sqrt(k)
    theta = ((A[:, idx] @ torch.linalg.solve_triangular(R, Om, upper=True)) ** 2).sum(1)
    (grad,) = torch.autograd.grad(theta, A, w.double())
    return {"theta": theta.detach(), "grad": grad}


def exact(case, seed):
    kind, d = case["kind"], case["d"]
    if kind == "rrqr":
        _, R = _pivoted_qr(_sketch_like(case["m"], d, seed).double(), case["tau"])
        return {"R": R, "rank": None, "perm": None}
    if kind == "train":
        return _exact_train(case, seed)
    if kind == "lstsq":
        A, b = _lstsq_inputs(case, seed)
        Q, R = torch.linalg.qr(A.double())
        return {"x": torch.linalg.solve_triangular(R, (Q.T @ b.double())[:, None], upper=True)[:, 0], "rank": None}
    n = case["n"]
    if kind in ("estimate_csr", "exact_csr"):
        csr = _csr(case, seed)
        At = _sketch_csr(csr, n, d, case["s"], case["m"])
        if kind == "estimate_csr":
            M = _small_factor(At, case["tau"], case["k"])
            theta = _csr_pair_norms(csr, case, M) if case["pairs"] else _csr_row_norms(csr, n, d, M)
        else:
            piv, _ = _pivoted_qr(At, case["tau"])
            theta = _csr_row_norms(csr, n, d, _leverage_factor(_csr_gram(csr, n, d), piv))
        return {"theta": theta, "rank": None, "perm": None}
    A = _dense(n, d, case["rank"], case["skew"], seed)
    if kind == "reference":                               # full column rank: any column order gives theta
        M = _leverage_factor(_gram(A), list(range(d)))
    else:
        At = _sketch_dense(A, case["s"], case["m"])
        if kind == "exact":
            M = _leverage_factor(_gram(A), _pivoted_qr(At, case["tau"])[0])
        else:
            M = _small_factor(At, case["tau"], case["k"])
    out = {"theta": _row_norms(A, M), "perm": None}
    if kind != "estimate" or case["wait"]:
        out["rank"] = None
    return out
