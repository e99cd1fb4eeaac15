"""Parity of the block tier for operands of any number of rows up to its limit: its shared
memory follows the rows (whole bitmap words, whole words of the first-level bitmap), with
columns beyond the sort tier's products, in both group sizes, flat and through a merge."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_matches, check_product, sp
from helpers import DT, MP_F32, OR_BOOL, PT_I64
from paper_1006_2183_gb300.gen import CSC

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


@pytest.mark.parametrize("m", [1, 31, 33, 1023, 1024, 1025, 8192, 20000, 32767, 32768])
@pytest.mark.parametrize("sr", [PT_I64, MP_F32, OR_BOOL])
def test_block_tier_rows(ctx, m, sr):
    rng = np.random.default_rng(0xB10C + m)

    def csc(rows, cols):
        ptr = np.concatenate(([0], np.cumsum([len(c) for c in cols]))).astype(np.int64)
        idx = np.concatenate(cols).astype(np.int32)
        v = rng.integers(0, 9, len(idx)) if sr != OR_BOOL else rng.random(len(idx)) < 0.9
        return CSC(rows, len(cols), ptr, idx, v.astype(DT[sr]))
    a = [np.sort(rng.choice(m, min(m, int(n)), replace=False)) for n in rng.integers(1, 40, 700)]
    a += [np.array([m - 1])] * 20 + [np.arange(m)] * 3   # the last row, and every row
    A = csc(m, a)
    b = [np.sort(rng.choice(700, n, replace=False)) for n in (8, 20, 60, 200, 699)]
    b += [np.arange(700, 720), np.array([3, 720, 721, 722]), np.arange(723), np.zeros(0, np.int64)]
    B = csc(len(a), b)
    R = check_product(ctx, A, B, sr, what=f"{m} rows")
    s = sp()
    dA, dB = s.Matrix.from_host(ctx, A, sr), s.Matrix.from_host(ctx, B, sr)
    assert_matches(s.spgemm_summa_blocked(ctx, dA, dB, 3, sr).to_host(), oracle.spgemm(A, B, sr), sr)
    assert R.nnz > 0
