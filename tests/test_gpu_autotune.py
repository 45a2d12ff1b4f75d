"""sscf_autotune reports the launch shape that it leaves in force.

At 216 molecules in FP64 the number of CTAs per tile taken by size (32 per SM over
54 occupied tiles, about 90) shares the pairs over the SMs far more evenly than 1,
2, 4 or 8 do, so it wins, and it is what later transforms run with.
"""
import pytest

from gpu_common import context, water

pytestmark = pytest.mark.gpu


def test_the_number_by_size_is_reported_where_it_wins():
    import torch
    s = water(216)
    ctx = context(s)
    ctx.set_thresholds(1e-3, 1e-2, 1e-8)
    ctx.guess()
    ctx.orthonormalise(0, max_pass=50)
    ctx.set_thresholds(1e-5, 1e-4, 1e-6)
    ctx.reset_charges()
    ctx.step()
    n_sm = torch.cuda.get_device_properties(0).multi_processor_count
    by_size = min(128, max(8, -(-32 * n_sm // 54)))
    v = ctx.autotune()
    ctx.close()
    assert v % 16 in (1, 2, 4, 8) and v // 16 == by_size
