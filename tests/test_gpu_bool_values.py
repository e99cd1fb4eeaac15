"""A boolean plan computes from the values that its operands hold when it is executed, not
from those of its making: all true, then some false, then all true again, in every tier."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_matches, sp
from helpers import OR_BOOL
from paper_1006_2183_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context(stream=torch.cuda.Stream())


def _values(rnd, nnz, seed):
    """False in two entries of three in the odd rounds."""
    return (np.random.default_rng(seed + rnd).integers(0, 3 if rnd % 2 else 1, nnz) == 0).astype(np.uint8)


def _operand(ctx, M, t):
    d = ctx.device
    return sp().Matrix.csc(ctx, M.m, M.n, torch.from_numpy(M.colptr).to(d), torch.from_numpy(M.rowidx).to(d), t, OR_BOOL)


# 1,024 rows: sort and block tiers; 65,536: sort tier, hash tables beyond 512 products
# (warp_max_flops 128) and slabs
CASES = [(10, 512), (16, 512), (16, 128)]


@pytest.mark.parametrize("scale,warp_max", CASES)
def test_replayed_batch(ctx, scale, warp_max):
    s = sp()
    mats = [gen.rmat(scale, 8, 0xB01, OR_BOOL), gen.erdos_renyi(300, 300, 3, 0xB02, OR_BOOL)]
    vals = [torch.ones(M.nnz, dtype=torch.uint8, device=ctx.device) for M in mats]
    ops = [_operand(ctx, M, v) for M, v in zip(mats, vals)]
    plan = s.spgemm_batch_plan(ctx, ops, ops, OR_BOOL, s.default_opts(warp_max_flops=warp_max))
    outs = plan.outputs()
    for rnd in range(4):
        now = [_values(rnd, M.nnz, 0xB03) for M in mats]
        with torch.cuda.stream(ctx.stream):
            for v, h in zip(vals, now):
                v.copy_(torch.from_numpy(h))
        plan.execute()
        ctx.stream.synchronize()
        for M, h, C in zip(mats, now, outs):
            N = M.with_vals(h)
            assert_matches(C.to_host(), oracle.spgemm(N, N, OR_BOOL), OR_BOOL, what=f"round {rnd}")


@pytest.mark.parametrize("scale,warp_max", CASES)
def test_numeric_of_a_plan(ctx, scale, warp_max):
    s = sp()
    M = gen.rmat(scale, 8, 0xB11, OR_BOOL)
    v = torch.ones(M.nnz, dtype=torch.uint8, device=ctx.device)
    A = _operand(ctx, M, v)
    plan = s.spgemm_plan(ctx, A, A, OR_BOOL, s.default_opts(warp_max_flops=warp_max))
    s.spgemm_symbolic(plan)
    for rnd in range(1, 4):
        h = _values(rnd, M.nnz, 0xB13)
        with torch.cuda.stream(ctx.stream):
            v.copy_(torch.from_numpy(h))
        N = M.with_vals(h)
        assert_matches(s.spgemm_numeric(plan).to_host(), oracle.spgemm(N, N, OR_BOOL), OR_BOOL, what=f"round {rnd}")
