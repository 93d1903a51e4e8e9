"""Performance cases of the library: what a tomography program has it do,
through the public calls of paper_1602_08604_gb300.lre.

Each case is one call on data shaped like the repository's own workloads:
per-basis outcome counts or shot records of GHZ, product and random
low-rank states, measured in all 3^n Pauli bases, and the projection of the
estimates made from them.  The inputs are drawn with torch from the seed
alone; exact() repeats the definition of each result in 64 bits (integer
Kronecker folds, one FP64 division, complex128 butterflies, a full
eigendecomposition), sharing nothing with the library.
"""
import math
import random

import torch

from paper_1602_08604_gb300 import lre

DEV = "cuda"

# ---------------------------------------------------------------- the cases


def listed():
    return [
        # one small experiment at a time (a four-qubit register, 81 settings):
        # the latency of a call
        dict(name="estimate n=4", op="estimate", n=4, kind="i32", state="ginibre", rank=2, shots=1000),
        # an odd size: one count tile row, 128 outcomes, 16-bit counts
        dict(name="estimate n=7", op="estimate", n=7, kind="i16", state="ginibre", rank=2, shots=1000),
        # a ten-qubit GHZ state with white noise, dense 32-bit counts (242 MB)
        dict(name="estimate n=10", op="estimate", n=10, kind="i32", state="ghz", noise=0.10, shots=1000),
        # the precision workload: many shots, 32-bit counts (8.7 GB)
        dict(name="estimate n=12", op="estimate", n=12, kind="i32", state="product", noise=0.05, shots=4096),
        # the largest: the full-size workload's state, counts and shot number
        # at the size that fits the device three times (26 GB of 16-bit counts)
        dict(name="estimate n=13", op="estimate", n=13, kind="i16", state="ghz", noise=0.05, shots=1000),
        # bases measured with unequal shot numbers: the FP64-weighted estimate
        dict(name="per-basis n=10", op="perbasis", n=10, kind="i32", state="product", noise=0.05, shots=1000),
        # shot records as the detectors give them, already on the device
        dict(name="records n=11", op="records", n=11, state="ghz", noise=0.05, shots=1000),
        # many small reconstructions at once, uneven sizes and shot numbers
        dict(name="batch 256", op="batch", count=256, lo=3, hi=9, mix=256),
        # the projection onto physical states of the first, third and fourth
        # workloads' estimates
        dict(name="project n=4", op="project", n=4, kind="i32", state="ginibre", rank=2, shots=1000),
        dict(name="project n=10", op="project", n=10, kind="i32", state="ghz", noise=0.10, shots=1000),
        dict(name="project n=12", op="project", n=12, kind="i32", state="product", noise=0.05, shots=4096),
        # end to end from pinned host shot records, results back in host memory
        dict(name="host records n=11", op="host", n=11, state="ghz", noise=0.05, shots=1000),
    ]


def _some_state(rng, n):
    """State options of a drawn case: any of the three families where it can be sampled quickly."""
    kind = rng.choice(["ghz", "product"] + (["ginibre"] if n <= 8 else []))
    if kind == "ginibre":
        return dict(state=kind, rank=rng.randint(1, 4))
    return dict(state=kind, noise=round(rng.uniform(0.02, 0.15), 3))


def draw(rng):
    op = rng.choice(["estimate", "estimate", "estimate", "estimate", "perbasis", "records", "batch", "project",
                     "project", "host"])
    shots = int(round(math.exp(rng.uniform(math.log(200), math.log(6000)))))
    if op == "batch":
        lo = rng.randint(2, 6)
        return dict(op=op, count=rng.randint(24, 300), lo=lo, hi=rng.randint(max(lo, 5), 9), mix=rng.randint(1, 10 ** 6))
    # the number of qubits is the logarithm of the size
    if op == "estimate":
        n = rng.randint(2, 13)
        kind = "i16" if n == 13 else rng.choice(["i16", "i32"])
        return dict(op=op, n=n, kind=kind, shots=min(shots, 2000) if n == 13 else shots, **_some_state(rng, n))
    if op == "perbasis":
        n = rng.randint(2, 11)
        return dict(op=op, n=n, kind=rng.choice(["i16", "i32"]), shots=shots, **_some_state(rng, n))
    if op == "project":
        n = rng.randint(2, 12)
        return dict(op=op, n=n, kind="i32", shots=max(shots, 500), **_some_state(rng, n))
    n = rng.randint(4, 11)  # records, host
    return dict(op=op, n=n, shots=shots, **_some_state(rng, n))


def _batch_members(case):
    """(n, shots, rank) of each instance of a batch: part of the case, not of the seed."""
    r = random.Random(case["mix"])
    out = []
    for _ in range(case["count"]):
        out.append((r.randint(case["lo"], case["hi"]), int(math.exp(r.uniform(math.log(500), math.log(10000)))),
                    r.randint(1, 4)))
    return out


def work(case):
    """Bytes a call cannot do without: its input read once, its outputs written once."""
    op = case["op"]
    if op == "batch":
        return {"bytes": sum(6 ** n * 4 + 4 ** n * 16 for n, _, _ in _batch_members(case)), "flops": 0}
    n = case["n"]
    if op == "project":
        return {"bytes": 4 ** n * 16 + 2 ** n * 8, "flops": 0}
    out = 4 ** n * 16  # theta (FP64) and rho (complex64)
    if op in ("records", "host"):
        return {"bytes": 3 ** n * case["shots"] * 2 + out, "flops": 0}
    es = 2 if case["kind"] == "i16" else 4
    return {"bytes": 6 ** n * es + (3 ** n * 8 if op == "perbasis" else 0) + out, "flops": 0}


# ---------------------------------------------------------------- inputs


def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _axes(n, b0, b1):
    """Axis digits [bases, n] of bases b0..b1 (0 X, 1 Y, 2 Z; qubit 1 first)."""
    b = torch.arange(b0, b1, device=DEV, dtype=torch.int64)
    return torch.stack([(b // 3 ** (n - 1 - q)) % 3 for q in range(n)], 1)


def _ghz_rows(n, noise, shots, b0, b1, g):
    """Outcome records [bases, shots] of (1 - noise) |GHZ><GHZ| + noise I/d."""
    a = _axes(n, b0, b1)
    w = 2 ** torch.arange(n - 1, -1, -1, device=DEV)
    zmask = ((a == 2) * w).sum(1, keepdim=True).int()
    ny = (a == 1).sum(1, keepdim=True)
    r = torch.randint(0, 2 ** n, (b1 - b0, shots), generator=g, device=DEV, dtype=torch.int32)
    coin = torch.randint(0, 2, (b1 - b0, shots), generator=g, device=DEV, dtype=torch.int32)
    e = torch.where(coin > 0, r | zmask, r & ~zmask)  # equal bits on the Z sites
    # no Z site: the parity of the outcome is fixed when the number of Y is even
    p = e ^ (e >> 8)
    p ^= p >> 4
    p ^= p >> 2
    p ^= p >> 1
    want = (ny % 4 == 2).int()
    fix = ((zmask == 0) & (ny % 2 == 0)).int()
    e ^= (((p & 1) ^ want) & fix)
    u = torch.rand((b1 - b0, shots), generator=g, device=DEV)
    return torch.where(u < noise, r, e)


def _product_rows(n, bloch, shots, b0, b1, g):
    """Outcome records of a product state with Bloch vectors [n, 3]."""
    a = _axes(n, b0, b1)
    rec = torch.zeros((b1 - b0, shots), dtype=torch.int32, device=DEV)
    for q in range(n):
        p1 = (0.5 * (1 - bloch[q][a[:, q]])).float()[:, None]  # probability of outcome 1
        rec += (torch.rand((b1 - b0, shots), generator=g, device=DEV) < p1).int() << (n - 1 - q)
    return rec


def _ginibre_probabilities(n, rank, g):
    """Born probabilities [3^n, 2^n] (FP64) of a random rank-`rank` mixture."""
    d = 2 ** n
    m = torch.randn((d, rank), generator=g, device=DEV, dtype=torch.complex128)
    x = m @ m.conj().T
    x = (x / torch.trace(x).real).reshape(d, d)
    # entries -> Pauli expectations, then letters -> (axis, outcome), qubit n first
    for _ in range(n):
        r, c = x.shape[-2] // 2, x.shape[-1] // 2
        v = x.reshape(-1, r, 2, c, 2)
        p = torch.stack([v[:, :, 0, :, 0] + v[:, :, 1, :, 1], v[:, :, 0, :, 1] + v[:, :, 1, :, 0],
                         1j * (v[:, :, 0, :, 1] - v[:, :, 1, :, 0]), v[:, :, 0, :, 0] - v[:, :, 1, :, 1]], 0)
        x = p.reshape(-1, r, c)  # this qubit's letter is the most significant so far
    t = x.real.reshape(-1)
    t = t.reshape(1, 4 ** n, 1)  # [axes of the qubits done][letters left][outcomes of the qubits done]
    for _ in range(n):
        A, L, O = t.shape
        v = t.reshape(A, L // 4, 4, O)
        i, k = v[:, :, :1], v[:, :, 1:]
        w = 0.5 * torch.stack([i + k, i - k], 3)  # [A, L/4, 3, 2, O]
        t = w.permute(2, 0, 1, 3, 4).reshape(3 * A, L // 4, 2 * O)
    return t.reshape(3 ** n, 2 ** n).clamp_min(0.0)


def _split_counts(p, shots, g):
    """Multinomial counts of each row of p (shots: number or per-row tensor) by binomial splitting."""
    B, d = p.shape
    c = torch.as_tensor(shots, device=DEV, dtype=torch.float32).expand(B).reshape(B, 1).contiguous()
    o = 1
    while o < d:
        m = p.reshape(B, o, 2, -1).sum(-1)
        q = (m[..., 0] / m.sum(-1).clamp_min(1e-300)).clamp(0.0, 1.0).float()
        first = torch.binomial(c, q, generator=g)
        c = torch.stack([first, c - first], 2).reshape(B, 2 * o)
        o *= 2
    return c


def _block(n, shots):
    return max(1, min(3 ** n, (1 << 27) // max(shots, 2 ** n)))


def _bloch(n, noise, g):
    v = torch.randn((n, 3), generator=g, device=DEV, dtype=torch.float64)
    return (1.0 - noise) * v / v.norm(dim=1, keepdim=True)


def _records(case, seed):
    """Shot records [3^n, shots] of a case (16-bit)."""
    n, shots, g = case["n"], case["shots"], _gen(seed)
    out = torch.empty((3 ** n, shots), dtype=torch.int16, device=DEV)
    if case["state"] == "ginibre":
        p = _ginibre_probabilities(n, case["rank"], g)
        out.copy_(torch.multinomial(p, shots, replacement=True, generator=g))
        return out
    bloch = _bloch(n, case["noise"], g)
    step = _block(n, shots)
    for b0 in range(0, 3 ** n, step):
        b1 = min(b0 + step, 3 ** n)
        rows = (_ghz_rows(n, case["noise"], shots, b0, b1, g) if case["state"] == "ghz"
                else _product_rows(n, bloch, shots, b0, b1, g))
        out[b0:b1] = rows
    return out


def _histogram(rec, n):
    nb = rec.shape[0]
    at = rec.long() + (torch.arange(nb, device=DEV) << n)[:, None]
    c = torch.zeros(nb << n, dtype=torch.int32, device=DEV)
    c.scatter_add_(0, at.reshape(-1), torch.ones((), dtype=torch.int32, device=DEV).expand(at.numel()))
    return c.reshape(nb, 1 << n)


def _counts(case, seed):
    """Dense counts [3^n, 2^n] of a case."""
    n, shots, g = case["n"], case["shots"], _gen(seed)
    dt = torch.int16 if case["kind"] == "i16" else torch.int32
    if case["state"] == "ginibre":
        return _split_counts(_ginibre_probabilities(n, case["rank"], g), shots, g).to(dt)
    bloch = _bloch(n, case["noise"], g)
    out = torch.empty((3 ** n, 2 ** n), dtype=dt, device=DEV)
    step = _block(n, shots)
    for b0 in range(0, 3 ** n, step):
        b1 = min(b0 + step, 3 ** n)
        rows = (_ghz_rows(n, case["noise"], shots, b0, b1, g) if case["state"] == "ghz"
                else _product_rows(n, bloch, shots, b0, b1, g))
        out[b0:b1] = _histogram(rows, n)
    return out


def _perbasis(case, seed):
    """Counts whose bases have unequal totals (a quarter of the shots of some lost), and the totals."""
    n, shots, g = case["n"], case["shots"], _gen(seed)
    c = _counts(case, seed)
    if case["state"] == "ginibre":  # keep each basis' counts up to a basis-dependent thinning
        keep = 1.0 - 0.25 * torch.rand((3 ** n, 1), generator=g, device=DEV)
        c = torch.binomial(c.float(), keep.expand(3 ** n, 2 ** n).contiguous(), generator=g).to(c.dtype)
    else:
        step = max(1, (1 << 27) >> n)
        for b0 in range(0, 3 ** n, step):
            blk = c[b0:b0 + step]
            keep = 1.0 - 0.25 * torch.rand((blk.shape[0], 1), generator=g, device=DEV)
            blk.copy_(torch.binomial(blk.float(), keep.expand(blk.shape).contiguous(), generator=g))
    c[:, 0] += 1  # no basis is empty
    return c, c.sum(1, dtype=torch.int64)


def _batch_counts(case, seed):
    g = _gen(seed)
    return [(_split_counts(_ginibre_probabilities(n, rank, g), shots, g).int().contiguous(), shots, n)
            for n, shots, rank in _batch_members(case)]


# ---------------------------------------------------------------- the calls

_ctx = None


def _context():
    """A program keeps one context."""
    global _ctx
    if _ctx is None:
        _ctx = lre.lre_create(0)
    return _ctx


def _outputs(n, **kw):
    return (torch.empty(4 ** n, dtype=torch.float64, **kw), torch.empty((2 ** n, 2 ** n), dtype=torch.complex64, **kw))


def prepare(case, seed):
    op, ctx = case["op"], _context()
    s = dict(op=op, ctx=ctx)
    if op == "batch":
        members = _batch_counts(case, seed)
        total = sum(4 ** n for _, _, n in members)
        s["theta"] = torch.empty(total, dtype=torch.float64, device=DEV)
        s["rho"] = torch.empty(total, dtype=torch.complex64, device=DEV)
        s["counts"] = [c for c, _, _ in members]
        s["items"] = (lre.lre_instance * len(members))()
        at = 0
        for k, (c, shots, n) in enumerate(members):
            s["items"][k] = lre.lre_instance(c.data_ptr(), lre.LRE_COUNTS_I32, n, shots,
                                             s["theta"][at:].data_ptr(), s["rho"][at:].data_ptr())
            at += 4 ** n
        torch.cuda.synchronize()
        lre.lre_batch_tune(ctx, s["items"])  # as the benchmark does: once for a batch
        return s
    n = s["n"] = case["n"]
    s["shots"] = case["shots"]
    if op == "estimate":
        s["counts"] = _counts(case, seed)
    elif op == "perbasis":
        s["counts"], s["shots"] = _perbasis(case, seed)
    elif op == "records":
        s["counts"] = _records(case, seed)
    elif op == "host":
        rec = _records(case, seed)
        s["counts"] = torch.empty(rec.shape, dtype=rec.dtype, pin_memory=True)
        s["counts"].copy_(rec)
        s["theta"], s["rho"] = _outputs(n, pin_memory=True)
        return s
    elif op == "project":
        s["mu"] = _assemble(_theta(_counts(case, seed), n, case["shots"]), n).to(torch.complex64)
        s["out"] = torch.empty_like(s["mu"])
        s["eig"] = torch.empty(2 ** n, dtype=torch.float64, device=DEV)
        return s
    s["theta"], s["rho"] = _outputs(n, device=DEV)
    return s


def run(s):
    op, ctx = s["op"], s["ctx"]
    if op == "batch":
        lre.lre_batch_run(ctx, s["items"])
    elif op == "project":
        lre.lre_project(ctx, s["mu"], s["n"], s["out"], eig_rho=s["eig"])
        return {"rho": s["out"], "eig": s["eig"]}
    elif op == "host":
        lre.lre_estimate_host(ctx, s["counts"], lre.LRE_HOST_RECORDS_U16, s["shots"], s["n"], s["theta"], s["rho"])
    elif op == "records":
        lre.lre_estimate(ctx, s["counts"], s["shots"], s["n"], s["theta"], s["rho"], kind=lre.LRE_SHOTS_U16)
    else:
        lre.lre_estimate(ctx, s["counts"], s["shots"], s["n"], s["theta"], s["rho"])
    return {"theta": s["theta"], "rho": s["rho"]}


# ---------------------------------------------------------------- 64-bit values


def _fold_qubit(x, A, O, C):
    """One qubit (the last axis digit and outcome bit) of [A][O][C]: letters I, X, Y, Z on top of C."""
    v = x.reshape(A // 3, 3, O // 2, 2, C)
    s, d = v[:, :, :, 0] + v[:, :, :, 1], v[:, :, :, 0] - v[:, :, :, 1]
    out = torch.empty((A // 3, O // 2, 4, C), dtype=x.dtype, device=x.device)
    out[:, :, 0] = s[:, 0] + s[:, 1] + s[:, 2]
    for k in range(3):
        out[:, :, 1 + k] = d[:, k]
    return out


def _sums(rows, n, dtype):
    """T^{(x)n} of rows(b0, b1), the [b1 - b0, 2^n] values of those bases; blocks of fixed top axes."""
    top = 0
    while 6 ** n // 3 ** top > 1 << 31:
        top += 1
    m, parts = n - top, []
    for b in range(3 ** top):
        x = rows(b * 3 ** m, (b + 1) * 3 ** m).to(dtype)
        A, O, C = 3 ** m, 2 ** n, 1
        for _ in range(m):
            x = _fold_qubit(x, A, O, C)
            A, O, C = A // 3, O // 2, 4 * C
        parts.append(x.reshape(1, O, C))
    x = torch.cat(parts, 0) if top else parts[0]
    A, O, C = 3 ** top, 2 ** top, 4 ** m
    for _ in range(top):
        x = _fold_qubit(x, A, O, C)
        A, O, C = A // 3, O // 2, 4 * C
    return x.reshape(-1)


def _weights(n):
    """3^k of every Pauli index, k its number of identity letters (FP64)."""
    w = torch.ones(1, dtype=torch.float64, device=DEV)
    one = torch.tensor([3.0, 1.0, 1.0, 1.0], dtype=torch.float64, device=DEV)
    for _ in range(n):
        w = (one[:, None] * w[None, :]).reshape(-1)
    return w


def _theta(counts, n, shots):
    dtype = torch.int32 if shots * 3 ** n < 2 ** 31 else torch.int64
    return _sums(lambda a, b: counts[a:b], n, dtype).double() / (shots * _weights(n))


def _theta_perbasis(counts, totals, n):
    return _sums(lambda a, b: counts[a:b].double() / totals[a:b, None].double(), n, torch.float64) / _weights(n)


def _assemble(theta, n):
    """rho = 2^-n sum_P t_P P in complex128."""
    x = theta.to(torch.complex128).reshape(-1, 1, 1)
    for _ in range(n):
        H, R, C = x.shape
        v = x.reshape(H // 4, 4, R, C)
        out = torch.empty((H // 4, 2, R, 2, C), dtype=x.dtype, device=x.device)
        out[:, 0, :, 0] = v[:, 0] + v[:, 3]
        out[:, 1, :, 1] = v[:, 0] - v[:, 3]
        out[:, 0, :, 1] = v[:, 1] - 1j * v[:, 2]
        out[:, 1, :, 0] = v[:, 1] + 1j * v[:, 2]
        x = out.reshape(H // 4, 2 * R, 2 * C)
    return x.reshape(2 ** n, 2 ** n) / 2 ** n


def _project(mu):
    """The closest density matrix in Frobenius norm, and its spectrum in decreasing order."""
    w, v = torch.linalg.eigh(mu.to(torch.complex128))
    lam = w.cpu().tolist()
    a, j, kept = 0.0, 0, len(lam)
    while lam[j] + a / kept < 0.0:
        a += lam[j]
        j += 1
        kept -= 1
    x = w.clone()
    x[:j] = 0.0
    x[j:] += a / kept
    return (v * x) @ v.conj().T, x.flip(0)


def exact(case, seed):
    op = case["op"]
    if op == "batch":
        theta, rho = [], []
        for c, shots, n in _batch_counts(case, seed):
            theta.append(_theta(c, n, shots))
            rho.append(_assemble(theta[-1], n).reshape(-1))
        return {"theta": torch.cat(theta), "rho": torch.cat(rho)}
    n = case["n"]
    if op == "project":
        mu = _assemble(_theta(_counts(case, seed), n, case["shots"]), n).to(torch.complex64)
        rho, eig = _project(mu)
        return {"rho": rho, "eig": eig}
    if op == "perbasis":
        counts, totals = _perbasis(case, seed)
        theta = _theta_perbasis(counts, totals, n)
    elif op in ("records", "host"):
        rec = _records(case, seed)
        step = _block(n, case["shots"])
        counts = torch.empty((3 ** n, 2 ** n), dtype=torch.int32, device=DEV)
        for b0 in range(0, 3 ** n, step):
            counts[b0:b0 + step] = _histogram(rec[b0:b0 + step], n)
        theta = _theta(counts, n, case["shots"])
    else:
        theta = _theta(_counts(case, seed), n, case["shots"])
    return {"theta": theta, "rho": _assemble(theta, n)}
