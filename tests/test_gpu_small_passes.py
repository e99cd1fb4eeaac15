"""The passes around the products at their own edges: the scan of the counts with its bins
and lists (one tile of 4,096 columns, two launches, and beyond 2,048 tiles three), and the
search for stored false values in byte arrays of any alignment."""
import numpy as np
import pytest

import oracle
from gpu_util import assert_matches, sp
from helpers import OR_BOOL, PT_I64
from paper_1006_2183_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


@pytest.mark.parametrize("n", [1, 1023, 4095, 4096, 4097, 12289, 2048 * 4096, 2048 * 4096 + 4097])
def test_counts_scan(ctx, n):
    """A(:, k) for one k per column, k in any order: C is a gather, written down directly."""
    import torch
    s = sp()
    rng = np.random.default_rng(n)
    lens = np.array([0, 1, 0, 3, 17, 40, 0, 70, 2, 150], np.int64)
    if n > 10 ** 6:
        lens = np.array([0, 1, 0, 3, 0, 2, 0, 1, 2, 17], np.int64)
    colptr = np.concatenate(([0], np.cumsum(lens)))
    rows = np.concatenate([np.sort(rng.choice(500, x, replace=False)) for x in lens]).astype(np.int32)
    vals = rng.integers(-9, 10, len(rows))
    k = rng.integers(0, len(lens), n).astype(np.int32)
    dev = ctx.device

    def up(x):
        return torch.from_numpy(np.ascontiguousarray(x)).to(dev)
    A = s.Matrix.csc(ctx, 500, len(lens), up(colptr), up(rows), up(vals), PT_I64)
    B = s.Matrix.csc(ctx, len(lens), n, torch.arange(n + 1, device=dev), up(k), None, PT_I64)
    C = s.spgemm_multiply(ctx, A, B, PT_I64).to_host()
    want = np.concatenate(([0], np.cumsum(lens[k])))
    np.testing.assert_array_equal(C.colptr, want)
    at = np.arange(want[-1]) - np.repeat(want[:-1], lens[k]) + np.repeat(colptr[:-1][k], lens[k])
    np.testing.assert_array_equal(C.rowidx, rows[at])
    np.testing.assert_array_equal(C.vals, vals[at])


@pytest.mark.parametrize("n", [1, 15, 16, 17, 47, 64, 1000])
def test_false_values_found_at_any_place(ctx, n):
    """One false among n values of A (a 1 x n row of entries), at every place of the array's
    ends, the array at every alignment."""
    import torch
    s = sp()
    dev = ctx.device
    colptr = torch.arange(n + 1, device=dev)
    rows = torch.zeros(n, dtype=torch.int32, device=dev)
    one = gen.identity(n, np.uint8)
    B = s.Matrix.from_host(ctx, one, OR_BOOL)
    for off in range(17):
        buf = torch.full((n + 40,), 7, dtype=torch.uint8, device=dev)
        buf[:off] = 0
        buf[off + n:] = 0   # outside the array: not to be seen
        v = buf[off:off + n]
        for at in sorted({-1, 0, n // 2, n - 1, min(15, n - 1), max(0, n - 16)}):
            v.fill_(7)
            if at >= 0:
                v[at] = 0
            A = s.Matrix.csc(ctx, 1, n, colptr, rows, v, OR_BOOL)
            C = s.spgemm_multiply(ctx, A, B, OR_BOOL)
            want = np.ones(n, np.uint8)
            if at >= 0:
                want[at] = 0
            np.testing.assert_array_equal(C.to_host().vals, want)
            if off in (0, 5):
                Cs = s.spgemm_summa_blocked(ctx, A, B, 2, OR_BOOL)
                np.testing.assert_array_equal(Cs.to_host().vals, want)


def test_many_reads_in_one_wait(ctx):
    """More operands without columns than one launch reads back: each one's pointer is checked."""
    import torch
    s = sp()
    dev = ctx.device
    empty = [s.Matrix.csc(ctx, 4, 0, torch.zeros(1, dtype=torch.int64, device=dev),
                          torch.zeros(0, dtype=torch.int32, device=dev), torch.zeros(0, dtype=torch.int64, device=dev),
                          PT_I64) for _ in range(21)]
    A = gen.erdos_renyi(4, 4, 2, 3, PT_I64)
    As = [s.Matrix.from_host(ctx, A, PT_I64) for _ in range(21)]
    for C in s.spgemm_batch(ctx, As, empty, PT_I64):
        assert C.shape() == (4, 0, 0)
    bad = s.Matrix.csc(ctx, 4, 0, torch.ones(1, dtype=torch.int64, device=dev),
                       torch.zeros(0, dtype=torch.int32, device=dev), None, PT_I64)
    fresh = [s.Matrix.csc(ctx, 4, 0, torch.zeros(1, dtype=torch.int64, device=dev),
                          torch.zeros(0, dtype=torch.int32, device=dev), None, PT_I64) for _ in range(20)]
    with pytest.raises(s.SpGEMMError):
        s.spgemm_batch(ctx, As, fresh[:13] + [bad] + fresh[13:], PT_I64)
    R = oracle.spgemm(A, A, PT_I64)
    assert_matches(s.spgemm_multiply(ctx, As[0], As[0], PT_I64).to_host(), R, PT_I64)
