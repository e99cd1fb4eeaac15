"""Parity of the sort tier where its keys run out of bits: operands of 2^22 - 1 rows (the
last with columns of 1024 products), one more, and the same at 2^23 .. 2^25 and 2^28 (where
no column fits and a thread or a table takes each), with rows 0 and m - 1 in use, columns
at every bin's edge (1, 16, 17 .. 1024, 1025 products), runs of equal rows that fill whole
columns, columns whose products come over many entries of B, and a DCSC A."""
import numpy as np
import pytest

import oracle
from gpu_util import sp
from helpers import DT, MP_F32, OR_BOOL, PT_F64, PT_I64
from paper_1006_2183_gb300.gen import CSC

pytestmark = pytest.mark.gpu
TARGETS = (1, 2, 15, 16, 17, 31, 32, 33, 64, 65, 127, 128, 129, 255, 256, 257, 400, 511, 512, 513, 700, 1023, 1024, 1025)


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


def _targets(m):
    """Columns of more than 1,024 products need row slabs, which 2^26 rows and more do not fit."""
    return [t for t in TARGETS if t <= 1024 or m < 2 ** 26]


def _operands(m, sr, seed):
    """A: columns 0..59 empty, 60..299 of 1..9 rows anywhere (0 and m - 1 often), 300..399 of
    1..3 of three rows, 400..599 of one row each.  B: per target a column of every style."""
    rng = np.random.default_rng(seed)
    cols = []
    for t in range(600):
        if t < 60:
            rows = np.zeros(0, np.int64)
        elif t < 300:
            rows = np.unique(np.concatenate((rng.integers(0, m, rng.integers(0, 8)), rng.choice([0, m - 1], 1))))
        elif t < 400:
            rows = rng.choice(np.array([0, m // 2, m - 1]), rng.integers(1, 4), replace=False)
        else:
            rows = np.array([m - 1 - t % 3])
        cols.append(np.sort(rows))
    lens = np.array([len(c) for c in cols])
    pool = {"any": np.arange(60, 300), "three": np.arange(300, 400), "single": np.arange(400, 600)}
    bcols = []
    for target in _targets(m):
        for style in pool:
            ks, f = [], 0
            # the style's columns first, then single rows until the target is met
            for k in np.concatenate((rng.permutation(pool[style]), rng.permutation(pool["any"]),
                                     rng.permutation(pool["single"]))):
                if f + lens[k] <= target and int(k) not in ks:
                    ks.append(int(k))
                    f += int(lens[k])
                if f == target:
                    break
            assert f == target
            if style == "three":
                ks += [int(k) for k in rng.choice(60, 40, replace=False)]
            bcols.append(np.sort(np.array(ks, np.int64)))

    def csc(rows, cs, s):
        r = np.random.default_rng(s)
        ptr = np.concatenate(([0], np.cumsum([len(c) for c in cs]))).astype(np.int64)
        idx = np.concatenate(cs).astype(np.int32)
        n = len(idx)
        v = {PT_F64: r.uniform(-1.0, 1.0, n), MP_F32: r.uniform(0.0, 4.0, n), OR_BOOL: r.random(n) < 0.8,
             PT_I64: r.integers(-3, 4, n)}[sr]
        return CSC(rows, len(cs), ptr, idx, v.astype(DT[sr]))
    return csc(m, cols, seed + 1), csc(600, bcols, seed + 2)


# |a b| <= 1 and at most 600 products (one per column of A) of random sign per entry: a sum whose terms cancel to
# 1e-3 still holds 600 * 2^-53 / 1e-3 < 1e-10 relative, so FP64 is compared with atol on the
# scale of the terms, 600 roundings of 2^-53 of sums below 600
ATOL = 600 * 600 * 2.0 ** -53


@pytest.mark.parametrize("sr", [PT_F64, MP_F32, OR_BOOL, PT_I64])
@pytest.mark.parametrize("m", [40000, 2 ** 22 - 1, 2 ** 22, 2 ** 23 - 1, 2 ** 23, 2 ** 24 - 1, 2 ** 24, 2 ** 25, 2 ** 28 - 1, 2 ** 28])
def test_sort_tier_at_the_keys_limits(ctx, m, sr):
    if m == 2 ** 28 and sr in (MP_F32, OR_BOOL):
        pytest.skip("the other tiers, covered by two semirings")
    A, B = _operands(m, sr, 0x50F7 + sr)
    fl = oracle.flops_per_col(A, B)
    assert sorted(set(fl.tolist())) == sorted(_targets(m))
    s = sp()
    dA, dB = s.Matrix.from_host(ctx, A, sr), s.Matrix.from_host(ctx, B, sr)
    R = oracle.spgemm(A, B, sr)
    outs = [s.spgemm_multiply(ctx, dA, dB, sr), s.spgemm_multiply(ctx, s.spgemm_mat_to_dcsc(ctx, dA), dB, sr),
            *s.spgemm_batch(ctx, [dA, dA], [dB, dB], sr)]
    for C in outs:
        C = C.to_host()
        np.testing.assert_array_equal(C.colptr, R.colptr)
        np.testing.assert_array_equal(C.rowidx, R.rowidx)
        if sr == PT_F64:
            np.testing.assert_allclose(C.vals, R.vals, rtol=0, atol=ATOL)
        else:
            np.testing.assert_array_equal(C.vals, R.vals)


@pytest.mark.parametrize("m", [40000, 2 ** 22, 2 ** 25])
@pytest.mark.parametrize("block_max", [-1, 600, 2048])
def test_tier_statistics_follow_the_thresholds(ctx, m, block_max):
    """Which kernel sorts a column does not show in the plan's statistics."""
    A, B = _operands(m, PT_I64, 0x51)
    fl = oracle.flops_per_col(A, B)
    lim = 1024 if block_max < 0 else block_max
    tier = np.where(fl == 0, 0, np.where(fl <= 512, 1, np.where(fl <= lim, 2, 3)))
    s = sp()
    dA, dB = s.Matrix.from_host(ctx, A, PT_I64), s.Matrix.from_host(ctx, B, PT_I64)
    p = s.spgemm_plan(ctx, dA, dB, PT_I64, s.default_opts(block_max_flops=block_max))
    s.spgemm_symbolic(p)
    want = np.bincount(tier, minlength=4).tolist()
    assert list(p.stats()["tiers"]) == want
    cols, flops = list(p.tier_stats()["cols"]), list(p.tier_stats()["flops"])
    assert cols == want and flops == [int(fl[tier == i].sum()) for i in range(4)]
