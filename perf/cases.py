"""What the speed of this library is measured on: products as its users call them.

Twelve listed cases, and drawn ones of the same ranges, go through the public entry
points of paper_1006_2183_gb300.spgemm.  Inputs are made on the GPU from the seed:
R-MAT (0.57, 0.19, 0.19, 0.05) with duplicates merged, Erdos-Renyi with a fixed number
of distinct rows per column, and the 7-point stencil of a 3D grid.  Values are
uniform(0, 1) (plus-times FP64, min-plus FP32), true (or-and bool) or uniform in
[-8, 8] (plus-times int64).

Kinds of case (key "kind"):
  flat      C = A*A, one spgemm_multiply
  summa     C = A*A on a virtual g x g grid, one spgemm_summa_blocked
  galerkin  R*(A*P) on an N^3 grid with 2x2x2 aggregates, two spgemm_multiply
  restrict  A*S^T and S*(A*S^T) of a graph contraction, S given in CSR
  tall      A times a tall-skinny matrix (a BFS step over many sources, or a sparse
            block of vectors) whose handle is new on every call
  batch     uneven independent products in one spgemm_batch
  replay    the values of a planned batch computed again, spgemm_batch_execute
  formats   P A P^T, A^T and the DCSC form of A
"""
from __future__ import annotations

import math
import random

import torch

from paper_1006_2183_gb300 import spgemm as sp

SEMIRING = {"pt64": sp.PLUS_TIMES_F64, "mp32": sp.MIN_PLUS_F32, "bool": sp.OR_AND_BOOL, "i64": sp.PLUS_TIMES_I64}
WIDTH = {"pt64": 8, "mp32": 4, "bool": 1, "i64": 8}
DEV = "cuda"


# ------------------------------------------------------------------ cases
def listed():
    return [
        # the smallest call: a small sparse matrix squared, where launches and waits count
        {"name": "er12_flat_pt64", "kind": "flat", "graph": "er", "n": 4096, "ef": 8, "sr": "pt64"},
        # the largest: the skewed graph squared (two-hop paths of a social network)
        {"name": "rmat20_flat_pt64", "kind": "flat", "graph": "rmat", "n": 1 << 20, "ef": 8, "sr": "pt64"},
        # an ordinary one: one relaxation of all-pairs shortest paths
        {"name": "rmat18_flat_mp32", "kind": "flat", "graph": "rmat", "n": 1 << 18, "ef": 8, "sr": "mp32"},
        # reachability within two hops, a vertex count that is no power of two
        {"name": "rmat_odd_flat_bool", "kind": "flat", "graph": "rmat", "n": 300007, "ef": 8, "sr": "bool"},
        # 2D Sparse SUMMA: hypersparse block products and the merge of their partials
        {"name": "rmat18_summa16_pt64", "kind": "summa", "graph": "rmat", "n": 1 << 18, "ef": 8, "g": 16, "sr": "pt64"},
        # the same on a ragged grid, blocks that the grid does not divide
        {"name": "rmat_odd_summa7_mp32", "kind": "summa", "graph": "rmat", "n": 100003, "ef": 8, "g": 7, "sr": "mp32"},
        # the set-up of one multigrid level: many short columns
        {"name": "galerkin128_pt64", "kind": "galerkin", "N": 128, "sr": "pt64"},
        # graph contraction: A S^T, then S (A S^T), the restriction kept by rows
        {"name": "restrict_rmat20_o4", "kind": "restrict", "n": 1 << 20, "ef": 8, "order": 4, "sr": "pt64"},
        # one BFS step from 128 sources, frontiers of 1 to 1000 vertices
        {"name": "bfs_rmat20_k128", "kind": "tall", "n": 1 << 20, "ef": 16, "k": 128, "lo": 1, "hi": 1000, "sr": "bool"},
        # many uneven products at once
        {"name": "batch20_i64", "kind": "batch", "count": 20, "lo": 10, "hi": 16, "mix": 4, "sr": "i64"},
        # the same structure again with new values: the numeric pass alone
        {"name": "replay20_i64", "kind": "replay", "count": 20, "lo": 10, "hi": 16, "mix": 4, "sr": "i64"},
        # what a graph goes through before its products: relabelling, transpose, DCSC
        {"name": "formats_rmat18_pt64", "kind": "formats", "n": 1 << 18, "ef": 16, "sr": "pt64"},
    ]


def _log_int(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(math.log2(lo), math.log2(hi))))


def draw(rng: random.Random):
    kind = rng.choice(["flat", "flat", "flat", "summa", "summa", "galerkin", "restrict", "tall", "tall", "batch",
                       "replay", "formats"])
    sr = rng.choice(["pt64", "pt64", "mp32", "bool", "i64"])
    if kind == "flat":
        if rng.random() < 0.35:
            return {"kind": kind, "graph": "er", "n": _log_int(rng, 1500, 1 << 20), "ef": rng.randint(2, 16), "sr": sr}
        return {"kind": kind, "graph": "rmat", "n": _log_int(rng, 4096, 1 << 19), "ef": rng.randint(4, 9), "sr": sr}
    if kind == "summa":
        return {"kind": kind, "graph": "rmat", "n": _log_int(rng, 1 << 14, 1 << 18), "ef": rng.randint(4, 8),
                "g": rng.choice([3, 4, 7, 8, 11, 16, 20]), "sr": sr}
    if kind == "galerkin":
        return {"kind": kind, "N": 2 * rng.randint(8, 72), "sr": "pt64"}
    if kind == "restrict":
        return {"kind": kind, "n": _log_int(rng, 1 << 14, 1 << 20), "ef": rng.randint(4, 8), "order": rng.randint(2, 8),
                "sr": sr}
    if kind == "tall":
        hi = _log_int(rng, 10, 20000)
        return {"kind": kind, "n": _log_int(rng, 1 << 15, 1 << 20), "ef": rng.randint(4, 16), "k": _log_int(rng, 8, 256),
                "lo": rng.choice([1, hi]), "hi": hi, "sr": sr}
    if kind in ("batch", "replay"):
        lo = rng.randint(8, 11)
        return {"kind": kind, "count": rng.randint(2, 21), "lo": lo, "hi": rng.randint(lo + 1, 15),
                "mix": rng.randint(1, 10 ** 6), "sr": sr}
    return {"kind": kind, "n": _log_int(rng, 1 << 13, 1 << 20), "ef": rng.randint(2, 16), "sr": sr}


# ------------------------------------------------------------------ inputs
def _gen(*numbers):
    g = torch.Generator(device=DEV)
    g.manual_seed(random.Random(str(numbers)).getrandbits(48))
    return g


def _values(sr, nnz, g):
    if sr == "pt64":
        return torch.rand(nnz, generator=g, device=DEV, dtype=torch.float64)
    if sr == "mp32":
        return torch.rand(nnz, generator=g, device=DEV, dtype=torch.float32)
    if sr == "bool":
        return torch.ones(nnz, device=DEV, dtype=torch.uint8)
    return torch.randint(-8, 9, (nnz,), generator=g, device=DEV, dtype=torch.int64)


def _compress(m, n, rows, cols):
    """CSC pattern of (rows, cols), duplicates merged, rows ascending."""
    key = torch.unique(cols * m + rows)
    colptr = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    colptr[1:] = torch.cumsum(torch.bincount(key // m, minlength=n), 0)
    return m, n, colptr, (key % m).to(torch.int32)


def _rmat(n, ef, g):
    scale, want = max(1, math.ceil(math.log2(n))), ef * n
    kept = []
    got = 0
    while got < want:
        e = want if n == 1 << scale else int(1.6 * (want - got)) + 1024
        r = torch.zeros(e, device=DEV, dtype=torch.int64)
        c = torch.zeros(e, device=DEV, dtype=torch.int64)
        for _ in range(scale):
            u = torch.rand(e, generator=g, device=DEV)
            r = (r << 1) | (u >= 0.76)
            c = (c << 1) | (((u >= 0.57) & (u < 0.76)) | (u >= 0.95))
        inside = (r < n) & (c < n)
        kept.append((r[inside], c[inside]))
        got += kept[-1][0].numel()
    return torch.cat([k[0] for k in kept])[:want], torch.cat([k[1] for k in kept])[:want]


def _er(n, ef, g):
    rows = torch.randint(0, n, (n, ef), generator=g, device=DEV).sort(1).values
    while ef > 1:
        bad = (rows[:, 1:] == rows[:, :-1]).any(1).nonzero().flatten()
        if bad.numel() == 0:
            break
        rows[bad] = torch.randint(0, n, (bad.numel(), ef), generator=g, device=DEV).sort(1).values
    return rows.flatten(), torch.repeat_interleave(torch.arange(n, device=DEV), ef)


def _graph(kind, n, ef, g, shift):
    """n x n pattern; vertex v of the graph that g draws is called (v + shift) mod n."""
    r, c = _er(n, ef, g) if kind == "er" else _rmat(n, ef, g)
    return _compress(n, n, (r + shift) % n, (c + shift) % n)


def _frontier(n, k, lo, hi, g, shift):
    """n x k with about 10^U(log10 lo, log10 hi) distinct rows per column."""
    u = torch.rand(k, generator=g, device=DEV, dtype=torch.float64)
    cnt = (10.0 ** (math.log10(lo) + u * (math.log10(hi) - math.log10(lo)))).round().long().clamp(1, n // 2)
    cols = torch.repeat_interleave(torch.arange(k, device=DEV), cnt)
    rows = torch.randint(0, n, (cols.numel(),), generator=g, device=DEV)
    return _compress(n, k, (rows + shift) % n, cols)


def _stencil(N, g):
    """7-point operator with varying coefficients on N^3 points, x fastest."""
    n = N ** 3
    i = torch.arange(n, device=DEV)
    rows, cols, vals = [i], [i], [torch.full((n,), 6.0, device=DEV, dtype=torch.float64)]
    for stride, coord in ((1, i % N), (N, (i // N) % N), (N * N, i // (N * N))):
        for d in (-1, 1):
            ok = ((coord + d >= 0) & (coord + d < N)).nonzero().flatten()
            rows.append(ok + d * stride)
            cols.append(ok)
            vals.append(-0.5 - torch.rand(ok.numel(), generator=g, device=DEV, dtype=torch.float64))
    r, c, v = torch.cat(rows), torch.cat(cols), torch.cat(vals)
    order = torch.argsort(c * n + r)
    colptr = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    colptr[1:] = torch.cumsum(torch.bincount(c, minlength=n), 0)
    return n, n, colptr, r[order].to(torch.int32), v[order]


def _aggregation(N):
    """P (N^3 x (N/2)^3) of 2x2x2 cells, and R = P^T: unit values."""
    M, n = N // 2, N ** 3
    i = torch.arange(n, device=DEV)
    agg = (i % N) // 2 + M * (((i // N) % N) // 2) + M * M * (i // (N * N) // 2)
    one = torch.ones(n, device=DEV, dtype=torch.float64)
    P = (n, M ** 3, torch.arange(0, n + 1, 8, device=DEV, dtype=torch.int64),
         torch.argsort(agg, stable=True).to(torch.int32), one)
    R = (M ** 3, n, torch.arange(n + 1, device=DEV, dtype=torch.int64), agg.to(torch.int32), one)
    return P, R


def _csc(ctx, mat, sr):
    m, n, cp, ir, v = mat
    return sp.Matrix.csc(ctx, m, n, cp, ir, v, SEMIRING[sr])


def _inputs(case, seed):
    """The operands of a case as (m, n, colptr, rowidx, values) on the device.  The graphs
    belong to the case, so that every seed gives results of the same sizes; the seed names
    their vertices (a rotation) and draws the values."""
    sr, kind = case["sr"], case["kind"]
    g = _gen("values", seed)

    def shift(n):
        return int(torch.randint(0, n, (1,), generator=g, device=DEV))

    def valued(pattern):
        return (*pattern, _values(sr, pattern[3].numel(), g))

    if kind == "galerkin":
        P, R = _aggregation(case["N"])
        return {"A": _stencil(case["N"], g), "P": P, "R": R}
    if kind in ("batch", "replay"):
        r = random.Random(case["mix"])
        pairs = []
        for i in range(case["count"]):
            n = int(2.0 ** r.uniform(case["lo"], case["hi"]))
            s = shift(n)
            pairs.append(tuple(valued(_graph(r.choice(["er", "rmat"]), n, r.choice([4, 8, 16, 32]),
                                             _gen(case["mix"], i, side), s)) for side in range(2)))
        return {"pairs": pairs}
    n, s = case["n"], shift(case["n"])
    x = {"A": valued(_graph(case.get("graph", "rmat"), n, case["ef"], _gen("graph", n, case["ef"]), s))}
    if kind == "restrict":
        agg = torch.randperm(n, generator=_gen("aggregates", n), device=DEV).roll(s) // case["order"]
        k = -(-n // case["order"])
        colptr = torch.zeros(k + 1, device=DEV, dtype=torch.int64)
        colptr[1:] = torch.cumsum(torch.bincount(agg, minlength=k), 0)
        one = torch.zeros if sr == "mp32" else torch.ones
        # S by rows is S^T by columns: n x k, one entry per vertex
        x["St"] = (n, k, colptr, torch.argsort(agg, stable=True).to(torch.int32),
                   one(n, device=DEV, dtype=sp.TORCH_DTYPE[SEMIRING[sr]]))
    elif kind == "tall":
        x["F"] = valued(_frontier(n, case["k"], case["lo"], case["hi"], _gen("frontier", n, case["k"]), s))
    elif kind == "formats":
        x["perm"] = torch.randperm(n, generator=g, device=DEV).to(torch.int32)
    return x


def prepare(case, seed):
    x, sr, kind = _inputs(case, seed), case["sr"], case["kind"]
    # a CUDA graph is replayed on a stream of its own; everything else on the current one
    ctx = sp.Context(stream=torch.cuda.Stream()) if kind == "replay" else sp.Context()
    s = {"case": case, "ctx": ctx}
    if kind in ("batch", "replay"):
        s["A"] = [_csc(ctx, a, sr) for a, _ in x["pairs"]]
        s["B"] = [_csc(ctx, b, sr) for _, b in x["pairs"]]
        if kind == "replay":
            s["plan"] = sp.spgemm_batch_plan(ctx, s["A"], s["B"], SEMIRING[sr])
            s["C"] = s["plan"].outputs()
        return s
    s["A"] = _csc(ctx, x["A"], sr)
    if kind == "galerkin":
        s["P"], s["R"] = _csc(ctx, x["P"], sr), _csc(ctx, x["R"], sr)
    elif kind == "restrict":
        m, n, cp, ir, v = x["St"]
        s["St"] = _csc(ctx, x["St"], sr)
        s["S"] = sp.Matrix.csr(ctx, n, m, cp, ir, v, SEMIRING[sr])
    elif kind == "tall":
        s["F"] = x["F"]
    elif kind == "formats":
        s["perm"] = x["perm"]
    return s


# ------------------------------------------------------------------ one pass
def _out(C):
    """C's arrays as zero-copy tensors that keep the handle alive."""
    arrays = list(C.export()[3:])
    for t in arrays:
        t.handle = C
    return arrays


def run(s):
    case, ctx = s["case"], s["ctx"]
    kind, sr = case["kind"], SEMIRING[case["sr"]]
    if kind == "flat":
        return _out(sp.spgemm_multiply(ctx, s["A"], s["A"], sr))
    if kind == "summa":
        return _out(sp.spgemm_summa_blocked(ctx, s["A"], s["A"], case["g"], sr))
    if kind == "galerkin":
        AP = sp.spgemm_multiply(ctx, s["A"], s["P"], sr)
        return _out(AP) + _out(sp.spgemm_multiply(ctx, s["R"], AP, sr))
    if kind == "restrict":
        ASt = sp.spgemm_multiply(ctx, s["A"], s["St"], sr)
        return _out(ASt) + _out(sp.spgemm_multiply(ctx, s["S"], ASt, sr))
    if kind == "tall":
        return _out(sp.spgemm_multiply(ctx, s["A"], _csc(ctx, s["F"], case["sr"]), sr))
    if kind == "batch":
        return [t for C in sp.spgemm_batch(ctx, s["A"], s["B"], sr) for t in _out(C)]
    if kind == "replay":
        ctx.stream.wait_stream(torch.cuda.current_stream())
        s["plan"].execute()
        torch.cuda.current_stream().wait_stream(ctx.stream)
        return [t for C in s["C"] for t in _out(C)]
    PAPt = sp.spgemm_mat_permute(ctx, s["A"], s["perm"], s["perm"])
    At = sp.spgemm_mat_transpose(ctx, s["A"])
    D = sp.spgemm_mat_to_dcsc(ctx, s["A"])
    nzc, jc, aux, chunk = D.export_dcsc()
    cp = D.export()[3]
    for t in (jc, aux, cp):
        t.handle = D
    return _out(PAPt) + _out(At) + [jc, aux, cp]


# ------------------------------------------------------------------ what a pass cannot do without
def _csc_bytes(n, nnz, w):
    return 8 * (n + 1) + (4 + w) * nnz


def work(case):
    """Operands read once and results written once; two operations per multiply."""
    s, w = prepare(case, 0), WIDTH[case["sr"]]
    ctx, sr, kind = s["ctx"], SEMIRING[case["sr"]], case["kind"]

    def product(A, B):
        plan = sp.spgemm_plan(ctx, A, B, sr)
        nnz = sp.spgemm_symbolic(plan)
        return {"nnz": nnz, "flops": plan.stats()["flops"]}

    def size(M):
        _, n, nnz = M.shape()
        return _csc_bytes(n, nnz, w)

    if kind in ("flat", "summa"):
        r = product(s["A"], s["A"])
        return {"bytes": size(s["A"]) + _csc_bytes(case["n"], r["nnz"], w), "flops": 2 * r["flops"]}
    if kind in ("galerkin", "restrict"):
        right, left = (s["P"], s["R"]) if kind == "galerkin" else (s["St"], s["S"])
        r0 = product(s["A"], right)
        T = sp.spgemm_multiply(ctx, s["A"], right, sr)
        r1 = product(left, T)
        k = right.shape()[1]
        return {"bytes": size(s["A"]) + 2 * size(right) + 2 * size(T) + _csc_bytes(k, r1["nnz"], w),
                "flops": 2 * (r0["flops"] + r1["flops"])}
    if kind == "tall":
        # of A only the columns that the frontier meets, at most once each
        F = _csc(ctx, s["F"], case["sr"])
        r = product(s["A"], F)
        met = torch.unique(s["F"][3].long())
        cp = s["A"].export()[3]
        entries = int((cp[met + 1] - cp[met]).sum())
        return {"bytes": 16 * met.numel() + (4 + w) * entries + size(F) + _csc_bytes(case["k"], r["nnz"], w),
                "flops": 2 * r["flops"]}
    if kind in ("batch", "replay"):
        total = {"bytes": 0, "flops": 0}
        for A, B in zip(s["A"], s["B"]):
            r = product(A, B)
            n = B.shape()[1]
            total["bytes"] += size(A) + size(B) + _csc_bytes(n, r["nnz"], w)
            total["flops"] += 2 * r["flops"]
        return total
    nzc = int((s["A"].export()[3].diff() > 0).sum())
    return {"bytes": 2 * size(s["A"]) + 4 * case["n"] + 2 * size(s["A"]) + 8 * (case["n"] + 1) + 20 * nzc, "flops": 0}


# ------------------------------------------------------------------ the values in 64 bits
_CHUNK = 1 << 26     # products expanded at a time
_MOST = 1500000000   # products beyond which the plain form takes too long


def _exact_sum(slot, count, x, y):
    """Per slot the sum of x * y: products split without error (Dekker), their leading
    parts summed on a fixed grid without rounding, the rest beside them."""
    def halves(v):
        t = v * 134217729.0
        hi = t - (t - v)
        return hi, v - hi

    p = x * y
    xh, xl = halves(x)
    yh, yl = halves(y)
    err = ((xh * yh - p) + xh * yl + xl * yh) + xl * yl
    grid = 1.5 * 2.0 ** 22   # |p| < 2^21: adding and taking away rounds p to multiples of 2^-30
    top = (p + grid) - grid
    lead = torch.zeros(count, device=DEV, dtype=torch.float64).index_add_(0, slot, top)
    rest = torch.zeros(count, device=DEV, dtype=torch.float64).index_add_(0, slot, (p - top) + err)
    return lead + rest


def _plain_product(A, B, sr):
    """A*B by expanding, sorting and combining its products; None where there are too many."""
    m, n = A[0], B[1]
    alen = A[2].diff()
    per_entry = alen[B[3].long()]
    upto = torch.zeros(B[3].numel() + 1, device=DEV, dtype=torch.int64)
    upto[1:] = torch.cumsum(per_entry, 0)
    at_col = upto[B[2]]                     # products before each column of B
    if int(at_col[-1]) > _MOST:
        return None
    bcol = torch.repeat_interleave(torch.arange(n, device=DEV), B[2].diff())
    ends = at_col.cpu()
    rows, vals, counts, j = [], [], [], 0
    while j < n:
        e = max(j + 1, int(torch.searchsorted(ends, int(ends[j]) + _CHUNK, right=True)) - 1)
        t0, t1 = int(B[2][j]), int(B[2][e])
        cnt = per_entry[t0:t1]
        t = torch.repeat_interleave(torch.arange(t0, t1, device=DEV), cnt)
        pos = torch.arange(t.numel(), device=DEV) - (upto[t] - upto[t0]) + A[2][B[3].long()[t]]
        key, slot = torch.unique(bcol[t] * m + A[3].long()[pos], return_inverse=True)
        x, y = A[4][pos].double(), B[4][t].double()
        if sr == "pt64":
            vals.append(_exact_sum(slot, key.numel(), x, y))
        else:
            least = torch.full((key.numel(),), math.inf, device=DEV, dtype=torch.float64)
            vals.append(least.scatter_reduce_(0, slot, x + y, "amin"))
        rows.append((key % m).to(torch.int32))
        counts.append(torch.bincount(key // m - j, minlength=e - j))
        j = e
    colptr = torch.zeros(n + 1, device=DEV, dtype=torch.int64)
    colptr[1:] = torch.cumsum(torch.cat(counts), 0)
    return m, n, colptr, torch.cat(rows), torch.cat(vals)


def _transpose(A):
    m, n, cp, ir, v = A
    cols = torch.repeat_interleave(torch.arange(n, device=DEV), cp.diff())
    order = torch.argsort(ir.long() * n + cols)
    colptr = torch.zeros(m + 1, device=DEV, dtype=torch.int64)
    colptr[1:] = torch.cumsum(torch.bincount(ir.long(), minlength=m), 0)
    return n, m, colptr, cols[order].to(torch.int32), v[order]


def exact(case, seed):
    kind, sr = case["kind"], case["sr"]
    if sr not in ("pt64", "mp32") or kind == "formats":
        return None   # whole numbers, or values that are only moved
    x = _inputs(case, seed)
    if kind in ("flat", "summa"):
        products = [_plain_product(x["A"], x["A"], sr)]
    elif kind == "tall":
        products = [_plain_product(x["A"], x["F"], sr)]
    elif kind in ("batch", "replay"):
        products = [_plain_product(A, B, sr) for A, B in x["pairs"]]
    else:
        T = _plain_product(x["A"], x["P"] if kind == "galerkin" else x["St"], sr)
        products = [T, _plain_product(x["R"] if kind == "galerkin" else _transpose(x["St"]), T, sr)]
    if any(C is None for C in products):
        return None
    return [v for C in products for v in (None, None, C[4])]
