"""Columns that the sort tier can hold are sorted whatever warp_max_flops is: the option moves
them between the plan's statistics and, beyond the sort tier, between hash tables."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import assert_matches, sp
from helpers import PT_F64, PT_I64
from paper_1006_2183_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context()


@pytest.mark.parametrize("m", [500, 40000])
@pytest.mark.parametrize("warp_max,block_max", [(8, -1), (128, -1), (300, 600), (512, 512), (128, 64)])
def test_statistics_and_values(ctx, m, warp_max, block_max):
    s = sp()
    rng = np.random.default_rng(0x57)
    A = gen.erdos_renyi(m, 3000, 20, 0x57A, PT_I64)
    cols = [np.sort(rng.choice(3000, k, replace=False)) for k in (0, 1, 3, 6, 7, 15, 16, 25, 26, 51, 52, 80) * 5]
    B = gen.CSC(3000, len(cols), np.concatenate(([0], np.cumsum([len(c) for c in cols]))).astype(np.int64),
                np.concatenate(cols).astype(np.int32), np.ones(sum(map(len, cols)), np.int64))
    fl = oracle.flops_per_col(A, B)
    cap = np.minimum(fl, m)
    lim = max(warp_max, block_max if block_max >= 0 else 4096 if m <= 32768 else 1024)
    tier = np.where(fl == 0, 0, np.where((cap <= warp_max) | (fl <= 16), 1, np.where(cap <= lim, 2, 3)))
    want = np.bincount(tier, minlength=4).tolist()
    dA, dB = s.Matrix.from_host(ctx, A, PT_I64), s.Matrix.from_host(ctx, B, PT_I64)
    p = s.spgemm_plan(ctx, dA, dB, PT_I64, s.default_opts(warp_max_flops=warp_max, block_max_flops=block_max))
    s.spgemm_symbolic(p)
    assert list(p.stats()["tiers"]) == want
    assert list(p.tier_stats()["cols"]) == want
    assert list(p.tier_stats()["flops"]) == [int(fl[tier == i].sum()) for i in range(4)]
    assert_matches(s.spgemm_numeric(p).to_host(), oracle.spgemm(A, B, PT_I64), PT_I64)


def test_a_smaller_warp_max_does_not_leave_the_sort_tier(ctx):
    """Columns of 289 products, warp_max_flops 128 against 512."""
    s = sp()
    A = s.Matrix.from_host(ctx, gen.erdos_renyi(1 << 17, 1 << 17, 17, 0x57B, PT_F64), PT_F64)
    times = []
    for warp_max in (512, 128):
        best = float("inf")
        for rnd in range(8):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            s.spgemm_multiply(ctx, A, A, PT_F64, s.default_opts(warp_max_flops=warp_max))
            b.record()
            b.synchronize()
            if rnd > 2:
                best = min(best, a.elapsed_time(b))
        times.append(best)
    assert times[1] < 1.15 * times[0], times
