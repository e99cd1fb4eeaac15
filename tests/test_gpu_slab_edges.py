"""Parity of the slab tier's passes at their edges: min-plus columns just below, at and above
the entries that add up in shared memory (and the other semirings on the same columns), a
column whose B column has more entries than a batch, segments that begin and end inside an
aligned quad, A arrays that are not 16-byte aligned, a DCSC A, and slabs cut small."""
import numpy as np
import pytest

import oracle
from gpu_util import sp
from helpers import DT, MP_F32, OR_BOOL, PT_F64, PT_I64
from paper_1006_2183_gb300.gen import CSC

pytestmark = pytest.mark.gpu
M = 40000   # more rows than the block tier takes
# shared-memory accumulators of a min-plus slab over M rows: 113,152 bytes less the segments
# (14,464), bitmap and ranks (20 bytes per 128 rows, one group to spare), 4 bytes each
CAP = (113152 - (14464 + (M // 128 + 1) * 20 + 15) // 16 * 16) // 4


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


def _operands(sr):
    """A: 1,200 columns of 1..7 rows, then columns of long runs of rows.  B: columns that reach
    CAP - 1, CAP and CAP + 1 distinct rows from two runs, a column of 1,100 short entries, and
    columns of many overlapping runs."""
    rng = np.random.default_rng(0x51AB + sr)
    cols = [np.sort(rng.choice(M, rng.integers(1, 8), replace=False)) for _ in range(1200)]
    runs = [(0, CAP - 1), (0, CAP), (0, CAP + 1), (5, 5 + CAP // 2), (M - CAP, M), (1, 4002), (3, 4000), (7001, 11002)]
    for a, b in runs:
        cols.append(np.arange(a, b))
    for _ in range(12):
        cols.append(np.sort(rng.choice(M, 3001, replace=False)))
    first = 1200
    bcols = [[first], [first + 1], [first + 2], [first, first + 3], [first + 1, first + 4],
             list(range(0, 1100)) + [first + 5], [first + 5, first + 6, first + 7],
             [first + 8 + i for i in range(12)], [3, first + 9, first + 12]]

    def csc(rows, cs, seed):
        r = np.random.default_rng(seed)
        ptr = np.concatenate(([0], np.cumsum([len(c) for c in cs]))).astype(np.int64)
        idx = np.concatenate([np.asarray(c) for c in cs]).astype(np.int32)
        n = len(idx)
        v = {PT_F64: r.uniform(0.0, 1.0, n), MP_F32: r.uniform(-2.0, 4.0, n), OR_BOOL: r.random(n) < 0.9,
             PT_I64: r.integers(-2 ** 40, 2 ** 40, n)}[sr]
        return CSC(rows, len(cs), ptr, idx, v.astype(DT[sr]))
    return csc(M, cols, 1), csc(len(cols), bcols, 2)


@pytest.mark.parametrize("sr", [MP_F32, PT_I64, OR_BOOL, PT_F64])
def test_slab_edges(ctx, sr):
    import torch
    s = sp()
    A, B = _operands(sr)
    R = oracle.spgemm(A, B, sr)
    assert {CAP - 1, CAP, CAP + 1} <= set(np.diff(R.colptr).tolist())
    dA, dB = s.Matrix.from_host(ctx, A, sr), s.Matrix.from_host(ctx, B, sr)
    # A's arrays one element off their allocation: no aligned quads
    ir = torch.empty(A.nnz + 1, dtype=torch.int32, device=ctx.device)[1:]
    v = torch.empty(A.nnz + 1, dtype=s.TORCH_DTYPE[sr], device=ctx.device)[1:]
    ir.copy_(torch.from_numpy(A.rowidx))
    v.copy_(torch.from_numpy(A.vals))
    off = s.Matrix.csc(ctx, A.m, A.n, torch.from_numpy(A.colptr).to(ctx.device), ir, v, sr)
    small = s.default_opts(range_slab_rows=4096, block_max_flops=512, dense_part_flops=1024)
    for a, opts in ((dA, None), (off, None), (s.spgemm_mat_to_dcsc(ctx, dA), None), (dA, small), (off, small)):
        C = s.spgemm_multiply(ctx, a, dB, sr, opts).to_host()
        np.testing.assert_array_equal(C.colptr, R.colptr)
        np.testing.assert_array_equal(C.rowidx, R.rowidx)
        if sr == PT_F64:   # at most 1,101 positive terms per entry: each addition rounds once
            np.testing.assert_allclose(C.vals, R.vals, rtol=1102 * 2.0 ** -53)
        else:
            np.testing.assert_array_equal(C.vals, R.vals)
