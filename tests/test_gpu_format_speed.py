"""Conversions of matrices whose entries crowd on few rows or columns, or leave most columns
empty, take about as long as those of evenly filled ones of the same size: no pass leaves such
a column, row or run to one CTA or one counter.  The bounds are two to four times the time of the
even matrix."""
import pytest
import torch

from gpu_util import sp
from helpers import PT_F64

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


def _time(op):
    for _ in range(3):
        op()
    best = float("inf")
    for _ in range(7):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        op()
        b.record()
        b.synchronize()
        best = min(best, a.elapsed_time(b))
    return best


def _handle(ctx, m, n, colptr, rows):
    s = sp()
    v = torch.ones(rows.numel(), device=ctx.device, dtype=torch.float64)
    return s.Matrix.csc(ctx, m, n, colptr.to(ctx.device), rows.to(ctx.device, torch.int32), v, PT_F64)


def _full(ctx, m, n):
    return _handle(ctx, m, n, torch.arange(n + 1) * m, torch.arange(m).repeat(n))


def _even(ctx, m, n, deg):
    """`deg` entries per column, spread over the rows."""
    rows = (torch.arange(n)[:, None] * 7919 + torch.arange(deg) * (m // deg)).remainder(m).sort(1).values
    return _handle(ctx, m, n, torch.arange(n + 1) * deg, rows.flatten())


def test_runs_of_empty_columns(ctx):
    n = 1 << 22
    at = torch.arange(1000) * (n // 1000)
    ptr = torch.zeros(n + 1, dtype=torch.int64)
    ptr[at + 1] = 1
    few, even = _handle(ctx, n, n, ptr.cumsum(0), at), _even(ctx, n, n, 1)
    t = sp().spgemm_mat_transpose
    assert _time(lambda: t(ctx, few)) < 4 * _time(lambda: t(ctx, even))


def test_few_long_columns(ctx):
    m = 1 << 20
    long, even = _full(ctx, m, 8), _full(ctx, 2896, 2896)
    p, q = (torch.randperm(k, device=ctx.device).to(torch.int32) for k in (m, 2896))
    t = sp().spgemm_mat_permute
    assert _time(lambda: t(ctx, long, p, None)) < 4 * _time(lambda: t(ctx, even, q, None))


def test_few_long_rows(ctx):
    long, even = _full(ctx, 8, 1 << 20), _full(ctx, 2896, 2896)
    t = sp().spgemm_mat_transpose
    assert _time(lambda: t(ctx, long)) < 2 * _time(lambda: t(ctx, even))


def test_permutation_of_empty_columns(ctx):
    """Against the same number of columns left in place: what is left is the check of the permutation."""
    n = 1 << 25
    at = torch.arange(1000) * (n // 1000)
    ptr = torch.zeros(n + 1, dtype=torch.int64)
    ptr[at + 1] = 1
    few = _handle(ctx, 1000, n, ptr.cumsum(0), torch.arange(1000))
    q, same = torch.randperm(n, device=ctx.device).to(torch.int32), torch.arange(n, device=ctx.device, dtype=torch.int32)
    t = sp().spgemm_mat_permute
    assert _time(lambda: t(ctx, few, None, q)) < 2.5 * _time(lambda: t(ctx, few, None, same))
