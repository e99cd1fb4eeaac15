"""Analysis of columns of B longer than the limit at which the whole CTA walks them:
lengths just at, below and above the limit and its rounds, several of them in one CTA,
with 1, 8 and 32 lanes per column (chosen by the mean length, set here by the number
of empty columns), against the oracle's features, flops and counts."""
import numpy as np
import pytest

import oracle
from gpu_util import check_product, sp
from helpers import PT_F64, PT_I64
from oracle import features as ofe
from paper_1006_2183_gb300.gen import CSC

pytestmark = pytest.mark.gpu
LENGTHS = (0, 1, 255, 256, 257, 1023, 1024, 1025, 1, 3000, 2049)


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


def _csc(m, cols, rng):
    ptr = np.concatenate(([0], np.cumsum([len(c) for c in cols]))).astype(np.int64)
    idx = np.concatenate(cols).astype(np.int32)
    return CSC(m, len(cols), ptr, idx, rng.uniform(0.0, 1.0, len(idx)))


@pytest.mark.parametrize("empty", [0, 200, 5000])
def test_hub_columns_analysis(ctx, empty):
    rng = np.random.default_rng(0x4B00 + empty)
    A = _csc(40000, [np.sort(rng.choice(40000, n, replace=False)) for n in rng.integers(0, 4, 3000)], rng)
    cols = [np.sort(rng.choice(3000, n, replace=False)) for n in LENGTHS * 3]
    cols += [np.zeros(0, np.int64)] * empty
    B = _csc(3000, cols, rng)
    s = sp()
    dA, dB = s.Matrix.from_host(ctx, A, PT_F64), s.Matrix.from_host(ctx, B, PT_F64)
    X, y = s.spgemm_predictor_features(ctx, dA, dB)
    d, fl, mx, pc = ofe.raw_features(A, B)
    np.testing.assert_allclose(X.cpu().numpy(), ofe.feature_vector(d, fl, mx, pc, A.m), rtol=2e-6, atol=2e-6)
    np.testing.assert_array_equal(y.cpu().numpy(), oracle.symbolic(A, B))
    assert s.spgemm_plan(ctx, dA, dB, PT_F64).stats()["flops"] == int(fl.sum())
    # a DCSC A (lookups through AUX, the A-column cache filled) gives the same product
    I = A.with_vals(np.arange(len(A.vals), dtype=np.int64) % 7 - 3)
    J = B.with_vals(np.arange(len(B.vals), dtype=np.int64) % 5 - 2)
    R = check_product(ctx, I, J, PT_I64, what="hub columns")
    dI, dJ = s.Matrix.from_host(ctx, I, PT_I64), s.Matrix.from_host(ctx, J, PT_I64)
    C = s.spgemm_multiply(ctx, s.spgemm_mat_to_dcsc(ctx, dI), dJ, PT_I64).to_host()
    np.testing.assert_array_equal(C.colptr, R.colptr)
    np.testing.assert_array_equal(C.rowidx, R.rowidx)
    np.testing.assert_array_equal(C.vals, R.vals)
