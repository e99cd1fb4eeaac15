"""Transpose and permutation with columns around the lengths from which a column is split over
several CTAs (16,384 entries for up to 2^20 keys, less for more, none up to 65,536 keys), alone and several at once,
down to a column that holds every key, with and without values."""
import numpy as np
import pytest
import torch

from gpu_util import sp
from helpers import DT, MP_F32, OR_BOOL, PT_F64
from oracle import formats as of
from paper_1006_2183_gb300.gen import CSC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


def _matrix(m, lengths, sr, seed):
    rng = np.random.default_rng(seed)
    cols = [np.sort(rng.permutation(m)[:n]) if n < m else np.arange(m) for n in lengths]
    ptr = np.concatenate(([0], np.cumsum([len(c) for c in cols]))).astype(np.int64)
    idx = np.concatenate(cols).astype(np.int32)
    return CSC(m, len(cols), ptr, idx, rng.integers(1, 200, len(idx)).astype(DT[sr]))


def _check(C, ref, vals=True):
    got = C.to_host() if vals else [t.cpu().numpy() for t in C.export()[3:5]]
    got = (got.colptr, got.rowidx, got.vals) if vals else got
    for g, w in zip(got, ref):
        np.testing.assert_array_equal(g, w)


@pytest.mark.parametrize("m,lengths,sr", [
    (100003, (0, 16383, 16384, 16385, 3, 100003, 40961, 513), PT_F64),
    (1 << 20, (1 << 20, 7, 16385, 1 << 20), MP_F32),
    (3000017, (5461, 5462, 0, 16384, 300000, 513), OR_BOOL),
    (2 ** 23 - 1, (2048, 2049, 8192, 8193, 500000, 1), PT_F64),
    (40000, (16385,), MP_F32),
    (65536, (65536, 16385), PT_F64),      # no column is split yet
    (65537, (65537, 16385), PT_F64),
])
def test_long_columns(ctx, m, lengths, sr):
    s = sp()
    A = _matrix(m, lengths, sr, 0x10E + m)
    rng = np.random.default_rng(8)
    p, q = rng.permutation(A.m).astype(np.int32), rng.permutation(A.n).astype(np.int32)
    dp, dq = torch.from_numpy(p).to(ctx.device), torch.from_numpy(q).to(ctx.device)
    back = (A.colptr, A.rowidx, A.vals)
    moved = of.permute(A.m, A.n, A.colptr, A.rowidx, A.vals, p, q)[:3]
    dA = s.Matrix.from_host(ctx, A, sr)
    T = s.spgemm_mat_transpose(ctx, dA)
    _check(T, of.transpose(A.m, A.n, A.colptr, A.rowidx, A.vals)[:3])
    _check(s.spgemm_mat_transpose(ctx, T), back)
    _check(s.spgemm_mat_permute(ctx, dA, dp, dq), moved)
    pattern = s.Matrix.csc(ctx, A.m, A.n, *(torch.from_numpy(x).to(ctx.device) for x in back[:2]), None, sr)
    _check(s.spgemm_mat_transpose(ctx, s.spgemm_mat_transpose(ctx, pattern)), back, vals=False)
    _check(s.spgemm_mat_permute(ctx, pattern, dp, dq), moved, vals=False)
