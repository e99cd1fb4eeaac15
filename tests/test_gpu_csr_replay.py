"""A replayed batch reads the current values of CSR operands too (they are converted once, with
the plan), a pattern-only one among them."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_matches, sp
from helpers import DT, MP_F32, OR_BOOL, PT_F64, PT_I64
from paper_1006_2183_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("sr", [PT_F64, MP_F32, OR_BOOL, PT_I64])
@pytest.mark.parametrize("own_stream", [False, True])
def test_csr_operands(sr, own_stream):
    s = sp()
    ctx = s.Context(stream=torch.cuda.Stream()) if own_stream else s.Context()
    d = ctx.device
    M = gen.rmat(11, 8, 0xC52, sr)      # stored by rows: the matrix itself is M^T
    v = torch.from_numpy(M.vals.copy()).to(d)
    A = s.Matrix.csr(ctx, M.n, M.m, torch.from_numpy(M.colptr).to(d), torch.from_numpy(M.rowidx).to(d), v, sr)
    ones = np.ones(M.nnz) if sr != MP_F32 else np.zeros(M.nnz)
    Q = s.Matrix.csr(ctx, M.n, M.m, torch.from_numpy(M.colptr).to(d), torch.from_numpy(M.rowidx).to(d), None, sr)
    B = gen.rmat(11, 4, 0xC53, sr)
    dB = s.Matrix.from_host(ctx, B, sr)
    plan = s.spgemm_batch_plan(ctx, [A, dB, Q], [dB, A, A], sr)
    outs = plan.outputs()
    rng = np.random.default_rng(5)
    Qt = gen.transpose_host(M.with_vals(ones.astype(DT[sr])))
    for rnd in range(3):
        now = rng.integers(0, 5, M.nnz).astype(DT[sr]) if rnd else M.vals
        torch.cuda.synchronize()
        v.copy_(torch.from_numpy(now))
        torch.cuda.synchronize()
        plan.execute()
        ctx.stream.synchronize()
        At = gen.transpose_host(M.with_vals(now))
        for C, (X, Y) in zip(outs, [(At, B), (B, At), (Qt, At)]):
            assert_matches(C.to_host(), oracle.spgemm(X, Y, sr), sr, what=f"round {rnd}")
