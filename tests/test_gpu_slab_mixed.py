"""Long columns of a batch whose operands differ in what the slab tier can read in aligned quads:
each product takes the form that its own A allows."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_matches, sp
from helpers import MP_F32, OR_BOOL, PT_F64, PT_I64
from paper_1006_2183_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


def _shifted(ctx, M, sr):
    """M's arrays one element past an aligned address."""
    d = ctx.device

    def place(x):
        t = torch.empty(x.size + 1, dtype=torch.from_numpy(x).dtype, device=d)[1:]
        return t.copy_(torch.from_numpy(x))

    return sp().Matrix.csc(ctx, M.m, M.n, torch.from_numpy(M.colptr).to(d), place(M.rowidx), place(M.vals), sr)


def _operands(ctx, sr):
    s = sp()
    mats = [gen.rmat(16, 8, 0x3A1 + i, sr) for i in range(3)] + [gen.erdos_renyi(300, 300, 3, 0x3A4, sr)]
    if sr == OR_BOOL:   # some false values: the products are evaluated
        mats = [M.with_vals((np.arange(M.nnz) % 5 != 0).astype(np.uint8)) for M in mats]
    A = [s.Matrix.from_host(ctx, mats[0], sr), _shifted(ctx, mats[1], sr),
         s.spgemm_mat_to_dcsc(ctx, s.Matrix.from_host(ctx, mats[2], sr)), _shifted(ctx, mats[3], sr)]
    return mats, A, [s.Matrix.from_host(ctx, M, sr) for M in mats]


@pytest.mark.parametrize("sr", [PT_F64, MP_F32, OR_BOOL, PT_I64])
@pytest.mark.parametrize("which", [(0, 1, 2, 3), (1, 2), (0, 3)])
def test_mixed_batch(ctx, sr, which):
    mats, A, B = _operands(ctx, sr)
    Cs = sp().spgemm_batch(ctx, [A[i] for i in which], [B[i] for i in which], sr)
    for i, C in zip(which, Cs):
        assert_matches(C.to_host(), oracle.spgemm(mats[i], mats[i], sr), sr, what=f"product {i}")


def test_slabs_over_columns_with_gaps(ctx):
    """The merge of SUMMA partials written into bounded slots, 65,536 rows to a block."""
    s = sp()
    M = gen.rmat(17, 4, 0x3A6, MP_F32)
    dM = s.Matrix.from_host(ctx, M, MP_F32)
    C = s.spgemm_summa_blocked(ctx, dM, dM, 2, MP_F32)
    assert_matches(C.to_host(), oracle.spgemm(M, M, MP_F32), MP_F32)


def test_an_unaligned_operand_slows_no_other(ctx):
    s = sp()
    big, tiny = gen.rmat(18, 8, 0x3A5, OR_BOOL), gen.erdos_renyi(300, 300, 3, 0x3A4, OR_BOOL)
    dB, dT = s.Matrix.from_host(ctx, big, OR_BOOL), s.Matrix.from_host(ctx, tiny, OR_BOOL)
    times = []
    for T in (dT, _shifted(ctx, tiny, OR_BOOL)):
        best = float("inf")
        for rnd in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            s.spgemm_batch(ctx, [dB, T], [dB, dT], OR_BOOL)
            b.record()
            b.synchronize()
            if rnd > 2:
                best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] < 1.06 * times[0], times
