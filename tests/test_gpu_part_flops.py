"""dense_part_flops counts as the caller gives it in every semiring: the slabs of a plan, seen
through the memory that their records and row sets take, do not depend on the values' type."""
import pytest
import torch

from gpu_util import sp
from helpers import MP_F32, OR_BOOL, PT_F64, PT_I64
from paper_1006_2183_gb300 import gen

pytestmark = pytest.mark.gpu


def _requested():
    return torch.cuda.memory_stats()["requested_bytes.all.current"]


@pytest.mark.parametrize("opts", [{"dense_part_flops": 262144}, {"dense_part_flops": 32768},
                                  {"dense_part_flops": 32768, "range_slab_rows": 1 << 20},
                                  {"dense_part_flops": 4096}])
def test_slabs_follow_the_option(opts):
    s = sp()
    ctx = s.Context()

    def taken(sr):
        A = s.Matrix.from_host(ctx, gen.rmat(17, 8, 0xF10, sr), sr)
        torch.cuda.synchronize()
        before = _requested()
        plan = s.spgemm_plan(ctx, A, A, sr, s.default_opts(**opts))
        after = _requested()
        plan.close()
        return after - before

    sizes = [taken(sr) for sr in (PT_F64, PT_I64, OR_BOOL, MP_F32)]
    assert sizes[0] > 0 and len(set(sizes)) == 1, sizes
