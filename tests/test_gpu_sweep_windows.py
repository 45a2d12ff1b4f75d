"""Sweeps in windows of colours, with several CTAs sharing a block's rows, equal the generic kernel.

In a cluster of 400 molecules the rows of a block make more runs than one CTA takes, so the
shares of a block, the flags that they raise and the fill between two windows all matter. FP32
agrees bit for bit; FP64 as in the sweeps of partly filled groups (1e-13: products may be
contracted differently).
"""
import numpy as np
import pytest

from gpu_common import context, water

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("window", [1, 3])
@pytest.mark.parametrize("prec", [0, 1])
def test_windows_of_shared_blocks_match_the_generic_kernel(window, prec):
    s = water(400)
    out = []
    for variant in (0, 1):
        ctx = context(s, precision=prec, apply_variant=variant, closure_mode=window)
        ctx.set_thresholds(1e-4, 1e-3, 1e-8)
        ctx.guess()
        ctx.orthonormalise(0, max_pass=1)
        ctx.orthonormalise(1, max_pass=1)
        ctx.build_fock()
        n_rot, _ = ctx.rotate_sweep()
        out.append((ctx.get_C(), n_rot))
        ctx.close()
    (C0, n0), (C1, n1) = out
    assert n0 == n1 > 0
    if prec:
        assert np.array_equal(C0, C1)
    else:
        assert np.abs(C0 - C1).max() <= 1e-13
