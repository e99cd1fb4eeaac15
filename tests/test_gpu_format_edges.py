"""Transpose, permutation and the block split at the edges of their passes: columns of 0 to
513 entries at every size class of the sort within columns, longer ones ranked through
bitmaps (one and several windows of 2^20 keys), runs of empty columns around the tiles of
2,048 entries, keys of 2^23 - 1 (the last that the sort holds) and beyond (radix passes)."""
import numpy as np
import pytest

from gpu_util import sp
from helpers import DT, MP_F32, OR_BOOL, PT_F64
from oracle import formats as of
from paper_1006_2183_gb300.gen import CSC

pytestmark = pytest.mark.gpu
LENGTHS = (0, 1, 2, 31, 32, 33, 64, 65, 128, 129, 256, 257, 511, 512, 513, 2047, 2048, 2049, 5000)


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


def _matrix(m, sr, seed, empties=0):
    rng = np.random.default_rng(seed)
    cols = []
    for n in rng.permutation(np.repeat(LENGTHS, 2)):
        n = min(int(n), m)
        rows = np.unique(np.concatenate((rng.integers(0, m, 2 * n), [0, m - 1]))) if n else np.zeros(0, np.int64)
        cols.append(np.sort(rng.choice(rows, min(n, len(rows)), replace=False)))
        cols += [np.zeros(0, np.int64)] * int(rng.integers(0, empties + 1))
    ptr = np.concatenate(([0], np.cumsum([len(c) for c in cols]))).astype(np.int64)
    idx = np.concatenate(cols).astype(np.int32)
    return CSC(m, len(cols), ptr, idx, rng.integers(1, 200, len(idx)).astype(DT[sr]))


def _same(C, ref):
    for got, want in zip((C.colptr, C.rowidx, C.vals), ref):
        np.testing.assert_array_equal(got, want)


@pytest.mark.parametrize("sr", [PT_F64, MP_F32, OR_BOOL])
@pytest.mark.parametrize("m,empties", [(70, 0), (5000, 4), (100003, 700), (3000017, 2), (2 ** 23 - 1, 0), (2 ** 23, 1)])
def test_transpose_and_permute(ctx, m, empties, sr):
    import torch
    s = sp()
    A = _matrix(m, sr, 0xF0 + m, empties)
    dA = s.Matrix.from_host(ctx, A, sr)
    T = s.spgemm_mat_transpose(ctx, dA)
    ref = of.transpose(A.m, A.n, A.colptr, A.rowidx, A.vals)
    _same(T.to_host(), ref[:3])
    _same(s.spgemm_mat_transpose(ctx, T).to_host(), (A.colptr, A.rowidx, A.vals))   # long keys now
    rng = np.random.default_rng(7)
    p, q = rng.permutation(A.m).astype(np.int32), rng.permutation(A.n).astype(np.int32)
    dp, dq = torch.from_numpy(p).to(ctx.device), torch.from_numpy(q).to(ctx.device)
    _same(s.spgemm_mat_permute(ctx, dA, dp, dq).to_host(), of.permute(A.m, A.n, A.colptr, A.rowidx, A.vals, p, q)[:3])
    i, j = np.arange(A.m, dtype=np.int32), np.arange(A.n, dtype=np.int32)
    _same(s.spgemm_mat_permute(ctx, dA, None, dq).to_host(), of.permute(A.m, A.n, A.colptr, A.rowidx, A.vals, i, q)[:3])
    _same(s.spgemm_mat_permute(ctx, dA, dp, None).to_host(), of.permute(A.m, A.n, A.colptr, A.rowidx, A.vals, p, j)[:3])


@pytest.mark.parametrize("g", [1, 3, 16])
def test_block_split_with_empty_columns(ctx, g):
    """The split's column numbers and AUX indexes, seen through the work of every block product."""
    s = sp()
    A = _matrix(9000, PT_F64, 0xF1, 300)
    rng = np.random.default_rng(9)
    n = 700
    B = CSC(A.n, n, np.arange(n + 1, dtype=np.int64), rng.integers(0, A.n, n).astype(np.int32), np.ones(n))
    got = s.spgemm_summa_block_flops(ctx, s.Matrix.from_host(ctx, A, PT_F64), s.Matrix.from_host(ctx, B, PT_F64), g)
    want = np.zeros((g, g, g), np.int64)
    kb, mb, nb = -(-A.n // g), -(-A.m // g), -(-n // g)
    for j in range(n):
        k = int(B.rowidx[j])
        rows = A.rowidx[A.colptr[k]:A.colptr[k + 1]]
        np.add.at(want, (k // kb, j // nb, rows // mb), 1)
    np.testing.assert_array_equal(got, want)
