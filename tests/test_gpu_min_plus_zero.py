"""Min-plus sums of negative zeros: (-0) + (-0) = -0 lies above every negative value of the
same entry, whichever tier adds the entry up and in whichever order."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import check_product, sp
from helpers import MP_F32
from paper_1006_2183_gb300 import gen

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    return sp().Context(stream=torch.cuda.Stream())


def _operands(m, k, deg, runs, seed):
    """A (m x k): columns of `deg` rows among few, so that entries meet; B (k x len(runs)):
    column j takes runs[j] columns of A.  Values: -0 and, rarely, negative."""
    rng = np.random.default_rng(seed)
    pool = np.sort(rng.choice(m, 4 * deg, replace=False))
    ar = np.concatenate([np.sort(rng.choice(pool, deg, replace=False)) for _ in range(k)]).astype(np.int32)
    br = np.concatenate([np.sort(rng.choice(k, r, replace=False)) for r in runs]).astype(np.int32)

    def vals(n):
        return np.where(rng.random(n) < 0.1, -rng.integers(1, 9, n), -0.0).astype(np.float32)

    A = gen.CSC(m, k, np.arange(k + 1, dtype=np.int64) * deg, ar, vals(ar.size))
    B = gen.CSC(k, len(runs), np.concatenate([[0], np.cumsum(runs)]).astype(np.int64), br, vals(br.size))
    return A, B


# products per column: sort tier (16 .. 1024), hash tables (warp_max_flops 16), block tier
# (1,000 rows) and slabs (8,000 products, 40,000 rows and more)
@pytest.mark.parametrize("m,opts", [
    (1000, {}),
    (40000, {}),
    (40000, {"warp_max_flops": 16, "block_max_flops": 4096}),
    (1 << 20, {"range_slab_rows": 1 << 20}),      # no room for sums in shared memory
])
def test_negative_zero_is_no_minimum(ctx, m, opts):
    A, B = _operands(m, 600, 40, [1, 2, 5, 10, 20, 60, 200, 500] * 4, 0x2E0)
    R = oracle.spgemm(A, B, MP_F32)
    assert (R.vals < 0).any() and (R.vals == 0).any()
    check_product(ctx, A, B, MP_F32, sp().default_opts(**opts), what=f"m={m} {opts}")
